"""The tcgen05 attention's device-side plan (which CTA takes which item, and how
many CTAs of a cluster share one) at the sizes where it changes shape, against
the oracle: attention within 2e-2, log-sum-exp within 2e-2 absolute."""
import pytest

import synth
from tests.test_gpu_attention import check_case, ssd  # noqa: F401 (ssd: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,B,heads,d,grid,prefix,cache", [
    # few live items: 4 CTAs of a cluster share each; the second sequence has
    # fewer key tiles (one) than CTAs, so some of them have no keys
    ("parts_without_keys", 2, (4, 4), 128, 24, 0, [24 * 20 + 5, 0]),
    # 64-row tiles, d = 64, each part one or two tiles
    ("short_parts", 1, (8, 8), 64, 16, 32, [200]),
    # 128-row tiles (GQA): two query tiles for the first sequence's 256 rows, one
    # for the second's last grid row; every other image complete
    ("tail_gqa", 8, (32, 8), 128, 32, 64, [64 + 1024] * 5 + [64 + 300, 64 + 1024, 64 + 31 * 32 + 4]),
    # 128 live items of at most 11 tiles: whole
    ("two_way", 8, (16, 16), 128, 24, 120, [120 + 72 * k for k in range(8)]),
    # 16 items of 17 tiles: 4 parts, of 4 tiles and one of 5
    ("four_short_parts", 1, (16, 16), 128, 32, 64, [64 + 975]),
    # 48 items of 16 and 17 tiles: 2 parts of 8 (4 would not have an SM each)
    ("two_parts_of_8", 3, (16, 16), 128, 32, 64, [64 + 940, 64 + 930, 64 + 960]),
    # 96 items of 24 tiles: 2 parts of 12 beyond one CTA per SM, where 23 stay whole
    ("two_parts_of_12", 6, (16, 16), 128, 40, 64, [64 + 1420] * 6),
    ("whole_below_12", 6, (16, 16), 128, 40, 64, [64 + 1320] * 6),
    # 160 ragged items of 2 to 26 tiles: the 128 longest take two CTAs each, the rest one
    ("longest_shared", 5, (32, 32), 64, 40, 0, [100, 400, 800, 1200, 1599]),
    ("longest_shared_block_plan", 40, (4, 4), 64, 40, 0, [1590 if k % 3 == 0 else 60 + 9 * k
                                                         for k in range(40)]),
    # more than 32 sequences: planned by the block (empty frontiers among them)
    ("block_plan", 40, (4, 4), 64, 16, 7, [7 + (37 * k) % 257 for k in range(40)]),
    # 3 and 20 query heads per KV head: tiles of 126 and 120 rows (42 and 6 drafts),
    # 63 of a 64-row tile with d = 64
    ("group_of_3", 3, (12, 4), 128, 24, 120, [120, 409, 120 + 23 * 24 + 1]),
    ("group_of_20", 2, (20, 1), 128, 12, 9, [9 + 30, 9 + 140]),
    ("group_of_3_64_rows", 4, (9, 3), 64, 10, 3, [3, 40, 77, 99]),
    # more than 128 query heads per KV head: the mma.sync kernel, splits merged
    # by its combine kernel
    ("group_of_150", 2, (150, 1), 64, 1, 300, [300, 301]),
    # more sequences than the plan holds: dealt in their order
    ("unplanned", 260, (1, 1), 64, 10, 3, [3 + (7 * k) % 101 for k in range(260)]),
    # five items per CTA of one to three key tiles, 64- and 128-row tiles
    ("many_items", 100, (16, 16), 64, 10, 3, [3 + (7 * k) % 101 for k in range(100)]),
    ("many_items_128", 24, (32, 8), 128, 16, 9, [9 + (31 * k) % 240 for k in range(24)]),
])
def test_plan_shapes(ssd, name, B, heads, d, grid, prefix, cache):  # noqa: F811
    c = synth.make_case(name, grid_h=max(grid, 3), grid_w=grid, prefix_len=prefix, cache_len=cache,
                        Hq=heads[0], Hkv=heads[1], d=d, V=64, seed=23, with_logits=False)
    assert c.B == B
    check_case(ssd, c)
