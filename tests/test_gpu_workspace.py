"""One workspace, sized for a program's longest array, serves its shorter
ones: at every length whose own choice of variant takes more than a longer
array's, the sort runs within the longer one's workspace (guards around it stay
intact) and gives the oracle's result."""
import numpy as np
import pytest

import inputs
import oracle

torch = pytest.importorskip("torch")
from gpu_util import from_dev, to_dev  # noqa: E402

from paper_1511_03404_gb300 import rs  # noqa: E402

pytestmark = pytest.mark.gpu
GUARD = 4096


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("dtype,pairs", [(np.uint32, False), (np.uint32, True),
                                         (np.uint64, False), (np.uint64, True)],
                         ids=["k32", "kv32", "k64", "kv64"])
def test_shorter_arrays_in_a_longer_ones_workspace(dtype, pairs, in_place):
    kb = np.dtype(dtype).itemsize
    vb = kb if pairs else 0
    stream = torch.cuda.current_stream().cuda_stream
    lengths = [2**e + q * 2**(e - 2) + d for e in range(12, 21) for q in range(4) for d in (0, 1)]
    need = {n: rs.rs_workspace_bytes(kb, vb, n, 0, 8 * kb)[1] for n in lengths + [250000, 300007]}
    asked = sorted(need)
    tried = 0
    for i, n in enumerate(asked):
        shorter = [x for x in asked[i + 1:] if need[x] < need[n]]
        for longer in sorted({min(shorter, key=need.get), shorter[0], shorter[-1]} if shorter else ()):
            tried += 1
            k = inputs.keys(dtype, "uniform", n)
            v = inputs.values(dtype, n) if pairs else None
            ws = torch.full((need[longer] + 2 * GUARD,), 0x5a, dtype=torch.uint8, device="cuda")
            dk = to_dev(k, torch)
            ka = torch.empty_like(dk)
            dv = to_dev(v, torch) if pairs else None
            va = torch.empty_like(dv) if pairs else None
            args = (kb, vb, dk.data_ptr(), dv.data_ptr() if pairs else None, ka.data_ptr(),
                    va.data_ptr() if pairs else None, n)
            at = ws.data_ptr() + GUARD
            for begin, end in ((0, 8 * kb), (0, 20)):
                dk.copy_(to_dev(k, torch))
                if pairs:
                    dv.copy_(to_dev(v, torch))
                if in_place:
                    st, alt = rs.rs_sort_in_place(*args, begin, end, at, need[longer], stream), 0
                else:
                    st, alt = rs.rs_sort(*args, begin, end, at, need[longer], stream)
                rs.check(st, (n, longer))
                rs.check(rs.rs_workspace_status(at, stream)[0])
                ek, ev = oracle.lsd_sort(k, v, begin_bit=begin, end_bit=end)
                assert np.array_equal(from_dev(ka if alt else dk, dtype), ek), (n, longer, end)
                assert not pairs or np.array_equal(from_dev(va if alt else dv, dtype), ev), (n, longer)
                assert bool((ws[:GUARD] == 0x5a).all()) and bool((ws[-GUARD:] == 0x5a).all())
    assert tried
