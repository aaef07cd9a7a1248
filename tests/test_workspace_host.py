"""Workspace sizes, on the host: what a tile shape asks for, and that a
workspace sized for one length serves every shorter one."""
import pytest
import torch

from paper_1511_03404_gb300 import rs

TYPES = [(4, 0), (4, 4), (8, 0), (8, 8)]


def up(x, a):
    return -(-x // a) * a


@pytest.mark.parametrize("kb,vb", TYPES)
def test_size_asked_by_a_tile_shape(kb, vb):
    """256 bytes, two tables of digit counts and, per pass, tile and digit, one
    32-bit word and two per 32 tiles (both counts rounded up to 4)."""
    for i in range(rs.rs_num_variants(kb, vb)):
        info = rs.rs_variant_info(kb, vb, i)
        if info["kind"] in (1, 4):  # held in shared memory
            continue
        radix = 1 << info["radix_bits"]
        for tiles in (1, 2, 3, 4, 5, 8, 9, 31, 33, 64, 65, 1000):
            n = tiles * info["threads"] * info["items"] - 1
            for bits in (8 * kb, 20, 3):
                passes = -(-bits // info["radix_bits"])
                table = passes * radix * 4
                words = passes * radix * 4 * (up(tiles, 4) + 2 * up(up(tiles, 32) // 32, 4))
                want = up(up(256 + table, 256) + table, 256) + up(words, 256)
                st, need = rs.rs_workspace_bytes(kb, vb, n, 0, bits, variant=i)
                assert st == rs.RS_OK and need == want, (i, tiles, bits)


def lengths():
    """The tuned bands' edges, what lies just past them, and between."""
    edges = sorted({2**e + q * 2**(e - 2) for e in range(4, 25) for q in range(4)})
    return sorted({n for e in edges for n in (e - 1, e, e + 1)} | {2, 250000, 300007})


@pytest.mark.skipif(torch.cuda.is_available(), reason="the pointers are not device memory")
@pytest.mark.parametrize("kb,vb", TYPES)
def test_a_longer_arrays_workspace_is_not_refused(kb, vb):
    """A sort that takes its workspace fails without a GPU (RS_ERR_CUDA); one
    that refuses it says RS_ERR_WORKSPACE."""
    at = [(1 + i) << 40 for i in range(5)]

    def status(n, bits, ws, ws_bytes):
        v, va = (at[2], at[3]) if vb else (None, None)
        return rs.rs_sort(kb, vb, at[0], v, at[1], va, n, 0, bits, ws, ws_bytes, None)[0]

    need = {n: rs.rs_workspace_bytes(kb, vb, n, 0, 8 * kb)[1] for n in lengths()}
    asked = sorted(need)
    more = 0
    for i, n in enumerate(asked):
        for longer in asked[i + 1:]:
            if need[longer] < need[n]:
                more += 1
                assert status(n, 8 * kb, at[4], need[longer]) == rs.RS_ERR_CUDA, (n, longer)
                assert status(n, 20, at[4], need[longer]) == rs.RS_ERR_CUDA, (n, longer)
        if need[n]:  # less than any length from n on is asked for
            least = min(need[x] for x in asked[i:])
            if least:
                assert status(n, 8 * kb, at[4], least // 2) == rs.RS_ERR_WORKSPACE, n
                assert status(n, 8 * kb, None, 0) == rs.RS_ERR_WORKSPACE, n
                assert status(n, 8 * kb, at[4] + 4, 2 * need[n]) == rs.RS_ERR_WORKSPACE, n
    assert more  # such lengths exist in the table
