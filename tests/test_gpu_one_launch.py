"""The one-launch form's barriers.  In the debug build all warps of a CTA but
the first read a barrier's outcome 20 us late (rs_fused.cuh, grid_barrier), so
that a word written too early after it takes warps out of the kernel and shows
as a wrong result.  Sizes of one tile, of less than a CTA a tile and of more
tiles than CTAs, inputs whose passes all move data, some or none, against the
oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
from gpu_util import sort_via_abi  # noqa: E402

from paper_1511_03404_gb300 import rs  # noqa: E402

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("dtype,pairs", [(np.uint32, False), (np.uint32, True),
                                         (np.uint64, False), (np.uint64, True)],
                         ids=["k32", "kv32", "k64", "kv64"])
def test_warps_that_read_the_barrier_late(dtype, pairs):
    if not rs.debug_library():
        pytest.skip("the late warps are in the debug build")
    kb = np.dtype(dtype).itemsize
    vb = kb if pairs else 0
    forms = [i for i in range(rs.rs_num_variants(kb, vb))
             if rs.rs_variant_info(kb, vb, i)["kind"] == 3]
    assert forms
    for i in forms:
        info = rs.rs_variant_info(kb, vb, i)
        tile = info["threads"] * info["items"]
        for n in (2, tile, 20 * tile + 3, 700 * tile + 5):
            v = inputs.values(dtype, n) if pairs else None
            for mask in (None, 0xff00, 0):
                k = inputs.keys(dtype, "uniform", n)
                k = k if mask is None else k & dtype(mask)
                gk, gv, _ = sort_via_abi(torch, k, v, variant=i)
                ek, ev = oracle.lsd_sort(k, v)
                assert np.array_equal(gk, ek), (i, n, mask)
                assert not pairs or np.array_equal(gv, ev), (i, n, mask)


def test_under_the_debug_build():
    if rs.debug_library():
        pytest.skip("already the debug build")
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.abspath(__file__), "-m", "gpu",
                        "-x", "-q", "-p", "no:cacheprovider", "-k", "late"], cwd=ROOT,
                       env=dict(os.environ, RS_LIBRARY="debug"), capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert "4 passed" in r.stdout and "skipped" not in r.stdout
