"""The digit passes rank with atomics whose order among equal digits is the
hardware's, check the order they got and repair it when it is not the input
order.  Here every warp's lanes take their keys in reverse (a test-only
knob), so that every repeated digit is out of turn and every tile needs the
repair; the result must still be the oracle's, bit for bit.  Keys of few
values make long runs of one digit, partial bit ranges take the slot-indexed
stage for keys too, and the sizes lie around one tile and around the groups
of 8 and 64 tiles of the look-back."""
import os
import subprocess
import sys

import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
from gpu_util import from_dev, sort_via_abi, to_dev  # noqa: E402

from paper_1511_03404_gb300 import rs  # noqa: E402

pytestmark = pytest.mark.gpu

TYPES = [(np.uint32, False), (np.uint32, True), (np.uint64, False), (np.uint64, True)]
TYPE_IDS = ["k32", "kv32", "k64", "kv64"]


def variants(kb, vb, kinds):
    out = [rs.rs_variant_info(kb, vb, i) | {"index": i} for i in range(rs.rs_num_variants(kb, vb))]
    return [v for v in out if v["kind"] in kinds]


def check(k, v, what, **kw):
    gk, gv, _ = sort_via_abi(torch, k, v, **kw)
    ek, ev = oracle.lsd_sort(k, v, begin_bit=kw.get("begin_bit", 0), end_bit=kw.get("end_bit"))
    assert np.array_equal(gk, ek), what
    assert v is None or np.array_equal(gv, ev), what


def merge_via_abi(k, v, kb, vb):
    n = k.shape[0]
    dk = to_dev(k, torch)
    ka = torch.empty_like(dk)
    dv = to_dev(v, torch) if vb else None
    va = torch.empty_like(dv) if vb else None
    st, need = rs.rs_merge_workspace_bytes(kb, vb, n)
    rs.check(st)
    ws = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
    st, alt = rs.rs_merge_sort(kb, vb, dk.data_ptr(), dv.data_ptr() if vb else None,
                               ka.data_ptr(), va.data_ptr() if vb else None, n, ws.data_ptr(),
                               ws.numel(), torch.cuda.current_stream().cuda_stream)
    rs.check(st)
    return (from_dev(ka if alt else dk, k.dtype).reshape(k.shape),
            from_dev(va if alt else dv, v.dtype) if vb else None)


class Repairs:
    """The count of tiles put in order and of sorts done again, which debug builds
    keep; in a release build it is taken to be what a test asks for."""

    def __init__(self):
        self.count = torch.zeros(1, dtype=torch.int32, device="cuda")
        st = rs.rs_debug_set(rs.RS_DEBUG_REPAIRS_PTR, self.count.data_ptr())
        assert st == (rs.RS_OK if rs.debug_library() else rs.RS_ERR_INVALID)

    def take(self):
        if not rs.debug_library():
            return 1 << 30
        n = int(self.count.item())
        self.count.zero_()
        return n


@pytest.fixture
def repairs():
    yield Repairs()
    torch.cuda.synchronize()
    rs.rs_debug_set(rs.RS_DEBUG_REPAIRS_PTR, 0)


@pytest.fixture
def mirrored():
    rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 1))
    yield
    rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 0))


@pytest.mark.parametrize("dtype,pairs", TYPES, ids=TYPE_IDS)
def test_out_of_turn_ranks_are_repaired(dtype, pairs, mirrored, repairs):
    kb = np.dtype(dtype).itemsize
    for var in variants(kb, kb if pairs else 0, (0, 1, 2, 3, 4)):
        tile = var["threads"] * var["items"]
        sizes = [tile - 1, tile, 3 * tile + 5]
        if var["max_n"] < 1 << 17:  # one CTA, one cluster: the work follows the length
            sizes += [2, 33, var["threads"] + 1, 5 * var["threads"] - 1,
                      8 * var["threads"] + 1, var["max_n"]]
        for n in sorted(s for s in sizes if s <= var["max_n"]):
            v = inputs.values(dtype, n) if pairs else None
            for name, k in (("uniform", inputs.keys(dtype, "uniform", n)),
                            ("few", inputs.keys(dtype, "uniform", n) & dtype(0x0303)),
                            ("sorted_desc", inputs.keys(dtype, "sorted_desc", n))):
                check(k, v, (name, n, var), variant=var["index"])
                # every digit has repeats in some warp from here on
                assert repairs.take() > 0 or name != "uniform" or n < 1000, (n, var)
            check(inputs.keys(dtype, "uniform", n), v, ("bits", n, var), variant=var["index"],
                  begin_bit=3, end_bit=17)
            assert repairs.take() > 0 or n < 1000, ("bits", n, var)


@pytest.mark.parametrize("dtype,pairs", TYPES, ids=TYPE_IDS)
def test_how_often_the_hardware_draws_out_of_turn(dtype, pairs, repairs):
    """Without the knob: the count of repairs is printed (-s), any is allowed."""
    if not rs.debug_library():
        pytest.skip("debug builds count")
    kb = np.dtype(dtype).itemsize
    for var in variants(kb, kb if pairs else 0, (0, 1, 2, 3, 4)):
        n = min(var["max_n"], 40 * var["threads"] * var["items"] + 3)
        check(inputs.keys(dtype, "gaussian", n), inputs.values(dtype, n) if pairs else None, var,
              variant=var["index"])
        print(f"k{kb} v{kb if pairs else 0} variant {var['index']}, {n} elements: "
              f"{repairs.take()} repairs")


@pytest.mark.parametrize("mirror", [0, 1])
@pytest.mark.parametrize("dtype,pairs", TYPES, ids=TYPE_IDS)
def test_tiles_around_the_look_back_levels(dtype, pairs, mirror, repairs):
    kb = np.dtype(dtype).itemsize
    try:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, mirror))
        for kind in (0, 2):
            var = min(variants(kb, kb if pairs else 0, (kind,)),
                      key=lambda x: x["threads"] * x["items"])
            tile = var["threads"] * var["items"]
            for tiles in (7, 8, 9, 63, 64, 65, 72, 129, 200):
                n = tiles * tile - 3
                v = inputs.values(dtype, n) if pairs else None
                check(inputs.keys(dtype, "gaussian", n), v, (n, var), variant=var["index"])
                assert not mirror or repairs.take() >= tiles, (n, var)  # in some pass each tile
                if not pairs and not mirror:
                    check(inputs.keys(dtype, "gaussian", n), v, (n, var, "bits"),
                          variant=var["index"], begin_bit=0, end_bit=20)
    finally:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 0))


@pytest.mark.parametrize("mirror", [0, 1])
@pytest.mark.parametrize("dtype,pairs", TYPES, ids=TYPE_IDS)
def test_segments_around_the_one_warp_and_one_cta_forms(dtype, pairs, mirror, repairs):
    """Empty, one-warp (up to 32), one-CTA (every number of items a thread, and
    the larger CTAs of medium ones) and tiled segments, more of them than one
    round of the planner takes."""
    rng = np.random.default_rng(7)
    lengths = [0, 1, 2, 31, 32, 33, 255, 256, 257, 1023, 1025, 2047, 2048, 2049, 3071,
               3072, 3073, 3841, 4096, 4097,
               8191, 8192, 8193, 12000, 0, 16383, 16384, 16385, 20479, 20480, 20481, 30011,
               70001]
    lengths += list(rng.integers(0, 70, 9000)) + [5, 0, 4096, 0]
    off = inputs.offsets_from_lengths(np.asarray(lengths, dtype=np.uint64))
    n = int(off[-1])
    kb = np.dtype(dtype).itemsize
    v = inputs.values(dtype, n) if pairs else None
    # segments of a CTA or more with keys enough for repeats in some warp
    certain = sum(int(x) >= 1000 for x in lengths)
    try:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, mirror))
        for k in (inputs.keys(dtype, "uniform", n), inputs.keys(dtype, "uniform", n) & dtype(0x303)):
            for begin, end in ((0, 8 * kb), (3, 20)):
                dk = to_dev(k, torch)
                dv = to_dev(v, torch) if pairs else None
                rs.segmented_sort(dk, to_dev(off, torch), dv, begin, end)
                ek, ev = oracle.segmented_sort(k, v, off, begin_bit=begin, end_bit=end)
                assert np.array_equal(from_dev(dk, dtype), ek), (begin, end)
                assert not pairs or np.array_equal(from_dev(dv, dtype), ev), (begin, end)
                assert not mirror or repairs.take() >= certain, (begin, end)
    finally:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 0))


@pytest.mark.parametrize("mirror", [0, 1])
@pytest.mark.parametrize("kb,vb", [(4, 0), (4, 4), (8, 0), (8, 8), (16, 0), (16, 8)])
def test_merge_tiles_by_bytes(kb, vb, mirror, repairs):
    """The merge sort's tiles: bytes that are the same in a whole tile are
    left out, few-valued ones repeat in every warp."""
    rng = np.random.default_rng(3)
    words = max(1, kb // 8)
    dt = np.uint32 if kb == 4 else np.uint64
    try:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, mirror))
        for n in (2, 33, 4095, 4096, 4097, 3 * 4096 + 77):
            for mask in (0, 0x30000, 0xff00ff00, None):
                k = rng.integers(0, np.iinfo(dt).max, (n, words), dtype=dt, endpoint=True)
                if mask is not None:
                    k &= dt(mask)
                k = k if words > 1 else k[:, 0]
                vdt = np.uint32 if vb == 4 else np.uint64
                v = np.arange(n, dtype=vdt) if vb else None
                gk, gv = merge_via_abi(k, v, kb, vb)
                ek, ev = oracle.sort_wide(k, v) if kb == 16 else oracle.lsd_sort(k, v)
                assert np.array_equal(gk, ek), (n, mask)
                assert not vb or np.array_equal(gv, ev), (n, mask)
                # equal keys are out of turn everywhere, distinct ones in some byte
                assert not mirror or repairs.take() >= n // 4096 or mask == 0, (n, mask)
    finally:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 0))


@pytest.mark.parametrize("dtype,pairs", TYPES, ids=TYPE_IDS)
def test_any_order_of_a_warps_draws_is_repaired(dtype, pairs, repairs):
    """A warp's keys of one digit in reverse, across its items: up to all the
    keys of a warp are out of place, and by as many places."""
    if not rs.debug_library():
        pytest.skip("the reversal is in the debug build")
    kb = np.dtype(dtype).itemsize
    try:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 2))
        for var in variants(kb, kb if pairs else 0, (0, 2, 3)):
            tile = var["threads"] * var["items"]
            for n in (33, tile - 1, 3 * tile + 5):
                v = inputs.values(dtype, n) if pairs else None
                for name, mask in (("uniform", None), ("few", 0x0303), ("two", 0x10001)):
                    k = inputs.keys(dtype, "uniform", n)
                    k = k if mask is None else k & dtype(mask)
                    check(k, v, (name, n, var), variant=var["index"])
                    check(k, v, (name, "bits", n, var), variant=var["index"], begin_bit=3,
                          end_bit=17)
                    assert repairs.take() > 0 or n < 1000, (name, n, var)
        rng = np.random.default_rng(5)
        off = inputs.offsets_from_lengths(np.asarray([30011, 70001, 20481, 5, 100000], np.uint64))
        n = int(off[-1])
        k = rng.integers(0, 4, n).astype(dtype)
        v = inputs.values(dtype, n) if pairs else None
        dk, dv = to_dev(k, torch), to_dev(v, torch) if pairs else None
        rs.segmented_sort(dk, to_dev(off, torch), dv)
        ek, ev = oracle.segmented_sort(k, v, off)
        assert np.array_equal(from_dev(dk, dtype), ek)
        assert not pairs or np.array_equal(from_dev(dv, dtype), ev)
    finally:
        rs.check(rs.rs_debug_set(rs.RS_DEBUG_MIRROR_LANES, 0))


def test_this_file_under_the_debug_build():
    """With the count of repairs, and the draws that only a debug build reverses."""
    if rs.debug_library():
        pytest.skip("already the debug build")
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.abspath(__file__), "-m", "gpu",
                        "-x", "-q", "-p", "no:cacheprovider", "-k", "not under_the_debug_build"],
                       env=dict(os.environ, RS_LIBRARY="debug"), capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "failed" not in r.stdout and "skipped" not in r.stdout
