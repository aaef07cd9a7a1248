"""The torch-level sorts on a stream that is not the current one: all of a call's
work, the copies back among it, runs on the stream it names, and the buffers
it allocates are not handed to the current stream while that work is pending."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
from gpu_util import from_dev, to_dev  # noqa: E402

from paper_1511_03404_gb300 import rs  # noqa: E402

pytestmark = pytest.mark.gpu
N = 300007
PENDING = int(2e8)  # clock cycles: about 0.1 s


def data():
    k = inputs.keys(np.uint32, "uniform", N)
    off = inputs.offsets_from_lengths(np.asarray([5000, 95007, 200000], np.uint64))
    return k, inputs.values(np.uint32, N), off


class Handle:
    """A stream of another library: no torch stream, only its handle."""

    def __init__(self, stream):
        self.cuda_stream = stream.cuda_stream


def call(segmented, k, off, v, stream):
    if segmented:
        rs.segmented_sort(k, off, v, 0, 20, stream=stream)  # three passes: ends in the alternates
    else:
        rs.sort(k, v, 0, 20, stream=stream, key_kind=rs.RS_KEY_UNSIGNED)


def expected(segmented):
    k, v, off = data()
    return (oracle.segmented_sort(k, v, off, begin_bit=0, end_bit=20) if segmented
            else oracle.lsd_sort(k, v, begin_bit=0, end_bit=20))


@pytest.mark.parametrize("handle_only", [False, True])
@pytest.mark.parametrize("segmented", [False, True])
def test_all_of_a_call_runs_on_its_stream(segmented, handle_only):
    k, v, off = (to_dev(x, torch) for x in data())
    side = torch.cuda.Stream()
    call(segmented, k.clone(), off, v.clone(), side)
    torch.cuda.synchronize()
    busy = torch.cuda.Event()
    torch.cuda._sleep(PENDING)  # the current stream is busy; nothing of the call may wait for it
    busy.record()
    call(segmented, k, off, v, Handle(side) if handle_only else side)
    with torch.cuda.stream(side):
        hk, hv = k.to("cpu", non_blocking=True), v.to("cpu", non_blocking=True)
    side.synchronize()
    assert not busy.query(), "the current stream's work ended before the sort's: nothing was tested"
    torch.cuda.synchronize()
    ek, ev = expected(segmented)
    assert np.array_equal(hk.numpy().view(np.uint32), ek)
    assert np.array_equal(hv.numpy().view(np.uint32), ev)


@pytest.mark.parametrize("segmented", [False, True])
def test_a_calls_buffers_are_its_streams(segmented, monkeypatch):
    k, v, off = (to_dev(x, torch) for x in data())
    name = "rs_segmented_sort" if segmented else "rs_sort_in_place"
    real, used = getattr(rs, name), []

    def spy(kb, vb, pk, pv, pka, pva, *rest, **kw):
        ws, ws_bytes = (rest[5], rest[6]) if segmented else (rest[3], rest[4])
        used.extend([(pka, 4 * N), (pva, 4 * N), (ws, ws_bytes)])
        return real(kb, vb, pk, pv, pka, pva, *rest, **kw)

    monkeypatch.setattr(rs, name, spy)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(PENDING)  # the sort is pending when the call returns
    call(segmented, k, off, v, side)
    assert len(used) == 3
    mine = [torch.empty(nbytes, dtype=torch.uint8, device="cuda") for _, nbytes in used * 3]
    for t in mine:
        t.fill_(0x5a)
    for at, nbytes in used:
        for t in mine:
            assert t.data_ptr() + t.numel() <= at or at + nbytes <= t.data_ptr()
    torch.cuda.synchronize()
    ek, ev = expected(segmented)
    assert np.array_equal(from_dev(k, np.uint32), ek)
    assert np.array_equal(from_dev(v, np.uint32), ev)


def test_sorts_of_several_streams_at_once():
    """Eight streams, each with its own buffers and workspace, enqueue sorts of
    every form side by side: one CTA, a cluster, one cooperative launch, ordinary
    and resident passes, segments; each result against the oracle."""
    streams = [torch.cuda.Stream() for _ in range(8)]
    jobs = []
    for i, n in enumerate([3000, 30000, 50000, 100003, 300007, 1 << 20, 3000017, 70001] * 3):
        dtype = (np.uint32, np.uint64)[i % 2]
        k, v = inputs.keys(dtype, "gaussian", n, seed=i + 1), inputs.values(dtype, n)
        jobs.append((i, k, v, to_dev(k, torch), to_dev(v, torch), i % 3 == 2))
    off = {n: np.asarray([0, n // 7, n // 2, n], np.uint64) for n in {j[1].size for j in jobs}}
    doff = {n: to_dev(o, torch) for n, o in off.items()}
    torch.cuda.synchronize()
    for i, k, v, dk, dv, segmented in jobs:
        if segmented:
            rs.segmented_sort(dk, doff[k.size], dv, 0, 20, stream=streams[i % 8])
        else:
            rs.sort(dk, dv, stream=streams[i % 8], key_kind=rs.RS_KEY_UNSIGNED)
    torch.cuda.synchronize()
    for i, k, v, dk, dv, segmented in jobs:
        ek, ev = (oracle.segmented_sort(k, v, off[k.size], begin_bit=0, end_bit=20) if segmented
                  else oracle.lsd_sort(k, v))
        assert np.array_equal(from_dev(dk, k.dtype), ek), (i, k.size)
        assert np.array_equal(from_dev(dv, k.dtype), ev), (i, k.size)
