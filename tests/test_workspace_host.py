"""Workspace sizes, on the host: what a tile shape asks for, and that a
workspace sized for one length serves every shorter one."""
import pytest

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
