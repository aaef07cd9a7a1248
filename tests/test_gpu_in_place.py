"""A sort whose result has to end where its input was starts, when its number
of passes is odd, from a copy that the counting kernel makes.  Bit ranges of
one, two and three passes, in every form that can end in the alternate
buffers, with the four arrays starting at 16-byte boundaries, all one element
past one, or each at its own offset (the copy then goes by elements), against
the oracle; nothing around the arrays may change."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
from gpu_util import from_dev, to_dev  # noqa: E402

from paper_1511_03404_gb300 import rs  # noqa: E402

pytestmark = pytest.mark.gpu

GUARD = 8


def forms(kb, vb):
    """One variant of each kind with global passes: the first compiled."""
    out = {}
    for i in range(rs.rs_num_variants(kb, vb)):
        out.setdefault(rs.rs_variant_info(kb, vb, i)["kind"], i)
    return [out[k] for k in (0, 2, 3) if k in out]


@pytest.mark.parametrize("dt", [np.uint32, np.uint64])
@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("offsets", [(0, 0, 0, 0), (1, 1, 1, 1), (0, 1, 3, 0)])
@pytest.mark.parametrize("bits", [(0, 20), (3, 8), (5, 21)])
def test_in_place(dt, pairs, offsets, bits):
    rng = np.random.default_rng(11)
    kb = np.dtype(dt).itemsize
    vb = kb if pairs else 0
    stream = torch.cuda.current_stream().cuda_stream
    for variant in forms(kb, vb):
        for n in (2, 33, 4099, 300007):
            def buffer(off):
                return to_dev(rng.integers(0, 2 ** 32, off + n + GUARD, dtype=dt), torch)
            bk, bv, bka, bva = (buffer(o) for o in offsets)
            before = [from_dev(b, dt) for b in (bk, bv)]
            k, v, ka, va = (b.data_ptr() + o * kb for b, o in zip((bk, bv, bka, bva), offsets))
            alts = [from_dev(b, dt) for b in (bka, bva)]
            ws = rs.workspace(kb, vb, n, *bits, variant=variant)
            rs.check(rs.rs_sort_in_place(kb, vb, k, v if pairs else None, ka,
                                         va if pairs else None, n, *bits, ws.data_ptr(),
                                         ws.numel(), stream, variant=variant))
            st, info = rs.rs_workspace_status(ws.data_ptr(), stream)
            rs.check(st)
            ok, ov = offsets[0], offsets[1]
            ek, ev = oracle.lsd_sort(before[0][ok:ok + n].copy(), before[1][ov:ov + n].copy(),
                                     begin_bit=bits[0], end_bit=bits[1])
            before[0][ok:ok + n] = ek
            if pairs:
                before[1][ov:ov + n] = ev
            what = (variant, n)
            if rs.debug_library():
                st, is_debug, site, index = rs.rs_debug_status()
                assert is_debug and st == rs.RS_OK, (what, site, index)
            assert np.array_equal(from_dev(bk, dt), before[0]), what
            assert np.array_equal(from_dev(bv, dt), before[1]), what
            for b, a, o in zip((bka, bva), alts, offsets[2:]):
                got = from_dev(b, dt)
                assert np.array_equal(got[:o], a[:o]) and np.array_equal(got[o + n:], a[o + n:]), what


@pytest.mark.parametrize("n", [5000, 300007, 3000001])
def test_in_place_captured(n):
    """Captured once, replayed on new inputs in the same buffers: the copy is
    part of the graph."""
    rng = np.random.default_rng(5)
    k = torch.empty(n, dtype=torch.int32, device="cuda")
    v, ka, va = (torch.empty_like(k) for _ in range(3))
    ws = rs.workspace(4, 4, n, 0, 20)
    side = torch.cuda.Stream()

    def sort():
        rs.check(rs.rs_sort_in_place(4, 4, k.data_ptr(), v.data_ptr(), ka.data_ptr(),
                                     va.data_ptr(), n, 0, 20, ws.data_ptr(), ws.numel(),
                                     torch.cuda.current_stream().cuda_stream))

    with torch.cuda.stream(side):
        k.zero_()
        v.zero_()
        sort()
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        sort()
    for _ in range(2):
        hk, hv = (rng.integers(0, 2 ** 32, n, dtype=np.uint32) for _ in range(2))
        k.copy_(to_dev(hk, torch))
        v.copy_(to_dev(hv, torch))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        ek, ev = oracle.lsd_sort(hk, hv, begin_bit=0, end_bit=20)
        assert np.array_equal(from_dev(k, np.uint32), ek)
        assert np.array_equal(from_dev(v, np.uint32), ev)


ORDERS = [(oracle.KEY_UNSIGNED, False), (oracle.KEY_UNSIGNED, True), (oracle.KEY_SIGNED, False),
          (oracle.KEY_FLOAT, True)]
ORDER_IDS = ["unsigned", "unsigned_desc", "signed", "float_desc"]


@pytest.mark.parametrize("dt", [np.uint32, np.uint64])
@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("kind,desc", ORDERS, ids=ORDER_IDS)
def test_in_place_orders_and_skipped_passes(dt, pairs, kind, desc):
    """Odd numbers of passes in every key order: the copy holds the keys as
    they came, the first pass that moves data transforms them.  Whole 32-bit keys
    at 7 bits a digit (five passes), where keys are staged themselves, and bit
    ranges of three; keys of which every pass moves data, some, or none."""
    rng = np.random.default_rng(13)
    kb = np.dtype(dt).itemsize
    vb = kb if pairs else 0
    stream = torch.cuda.current_stream().cuda_stream
    cases = [(i, bits) for i in forms(kb, vb) for bits in ((0, 20), (8 * kb - 20, 8 * kb))]
    cases += [(i, (0, 32)) for i in range(rs.rs_num_variants(kb, vb)) if kb == 4
              and rs.rs_variant_info(kb, vb, i)["radix_bits"] == 7]
    assert len(cases) == 6 + (kb == 4)
    for variant, bits in cases:
        info = rs.rs_variant_info(kb, vb, variant)
        assert -(-(bits[1] - bits[0]) // info["radix_bits"]) & 1
        for n in (33, 100003):
            for mask in (~0, 0xff << bits[0], 0x3 << (bits[1] - 2), 0):
                hk = rng.integers(0, 2 ** (8 * kb) - 1, n, dtype=dt, endpoint=True)
                hk &= dt(mask & (2 ** (8 * kb) - 1))
                hv = rng.integers(0, 2 ** 32, n, dtype=dt)
                k, v = to_dev(hk, torch), to_dev(hv, torch)
                ka, va = torch.zeros_like(k), torch.zeros_like(k)
                ws = rs.workspace(kb, vb, n, *bits, variant=variant)
                rs.check(rs.rs_sort_in_place(kb, vb, k.data_ptr(), v.data_ptr() if pairs else None,
                                             ka.data_ptr(), va.data_ptr() if pairs else None, n,
                                             *bits, ws.data_ptr(), ws.numel(), stream,
                                             variant=variant, key_kind=kind, descending=desc))
                st, s = rs.rs_workspace_stats(ws.data_ptr(), stream)
                rs.check(st)
                what = (variant, bits, n, mask)
                assert s["moved_mask"].bit_count() & 1, what  # from the copy back to the keys
                if kind == oracle.KEY_UNSIGNED and mask == 0:
                    assert s["moved_mask"] == 1, what
                ek, ev = oracle.ordered_sort(hk, hv, kind=kind, descending=desc,
                                             begin_bit=bits[0], end_bit=bits[1])
                assert np.array_equal(from_dev(k, dt), ek), what
                assert np.array_equal(from_dev(v, dt), ev if pairs else hv), what


@pytest.mark.parametrize("dt", [np.uint32, np.uint64])
@pytest.mark.parametrize("pairs", [False, True])
def test_the_record_counts_the_copy(dt, pairs):
    """rs_workspace_stats: n K for the histograms, 2 n (K + V) per moving pass,
    and n (K + 2 V) for the copy that an odd number of passes starts from."""
    kb = np.dtype(dt).itemsize
    vb = kb if pairs else 0
    n = 100003
    stream = torch.cuda.current_stream().cuda_stream
    hk = np.random.default_rng(3).integers(0, 2 ** 32, n, dtype=dt)
    for variant in forms(kb, vb):
        for end, passes in ((24, 3), (32, 4), (5, 1)):
            k = to_dev(hk, torch)
            v, ka, va = (torch.zeros_like(k) for _ in range(3))
            ws = rs.workspace(kb, vb, n, 0, end, variant=variant)
            rs.check(rs.rs_sort_in_place(kb, vb, k.data_ptr(), v.data_ptr() if pairs else None,
                                         ka.data_ptr(), va.data_ptr() if pairs else None, n, 0,
                                         end, ws.data_ptr(), ws.numel(), stream, variant=variant))
            st, s = rs.rs_workspace_stats(ws.data_ptr(), stream)
            rs.check(st)
            assert s["passes"] == passes and s["moved_mask"] == (1 << passes) - 1
            copy = n * (kb + 2 * vb) if passes & 1 else 0
            assert s["bytes"] == n * kb + copy + passes * 2 * n * (kb + vb), (variant, passes)


def test_in_place_under_the_debug_build():
    """The same calls with every store's index checked, those of the copy among them."""
    if rs.debug_library():
        pytest.skip("already the debug build")
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.abspath(__file__), "-m", "gpu",
                        "-x", "-q", "-p", "no:cacheprovider", "-k", "not under_the_debug_build"],
                       env=dict(os.environ, RS_LIBRARY="debug"), capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "failed" not in r.stdout
