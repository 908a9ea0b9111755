"""Cache slots past a sequence's keys (cache_len + n_drafts) belong to no one: whatever
they hold, NaN and infinities included, the attention's results are the same, bit
for bit, in every plan of both kernels."""
import numpy as np
import pytest

import synth
from tests.test_gpu_attention import check_case, run_attention, ssd  # noqa: F401 (ssd: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,B,heads,d,grid,prefix,cache", [
    # tcgen05: 64-row tiles whole, 4 CTAs per item, pairs of the longest, 128-row tiles
    ("whole", 8, (16, 16), 128, 24, 120, [120 + 72 * k for k in range(8)]),
    ("four_parts", 1, (8, 8), 64, 16, 32, [200]),
    ("four_parts_128", 1, (16, 16), 128, 32, 64, [64 + 975]),
    ("pairs", 5, (32, 32), 64, 40, 0, [100, 400, 800, 1200, 1599]),
    ("gqa", 8, (32, 8), 128, 32, 64, [64 + 1024] * 5 + [64 + 300, 64 + 1024, 64 + 31 * 32 + 4]),
    ("many_items", 100, (16, 16), 64, 10, 3, [3 + (7 * k) % 101 for k in range(100)]),
    # every number of keys in the last tile, one key and a full tile among them
    ("remainders", 65, (4, 4), 128, 9, 40, [40 + k for k in range(65)]),
    # mma.sync: one split, and splits merged by the combine kernel
    ("mma_sync", 3, (129, 1), 128, 1, 16, [16, 17, 18]),
    ("mma_sync_splits", 2, (150, 1), 64, 1, 300, [300, 301]),
    ("mma_sync_splits_128", 2, (256, 1), 128, 1, 700, [700, 702]),
])
def test_unused_slots_do_not_matter(ssd, name, B, heads, d, grid, prefix, cache):  # noqa: F811
    c = synth.make_case(name, grid_h=max(grid, 3), grid_w=grid, prefix_len=prefix, cache_len=cache,
                        Hq=heads[0], Hkv=heads[1], d=d, V=64, seed=29, with_logits=False)
    check_case(ssd, c)
    o, lse, nd, st = run_attention(ssd, c)
    assert st == 0
    rng = np.random.default_rng(29)
    junk = np.array([0x7fc0, 0xffc1, 0x7f80, 0xff80, 0x7f7f], np.uint16)  # NaN, inf, the largest
    for x in (c.k, c.v):
        for b in range(B):
            past = x[b, :, int(c.cache_len[b]) + int(nd[b]):]
            past[...] = rng.choice(junk, past.shape).astype(x.dtype)
    o2, lse2, _, st = run_attention(ssd, c)
    assert st == 0 and np.array_equal(o, o2) and np.array_equal(lse, lse2)
