"""The mma.sync attention (above 128 query heads per KV head) against the oracle:
one split and splits merged by the combine kernel, both head dimensions, a custom
scale, shuffled drafts, a bad draft position, and a workspace with old contents."""
import numpy as np
import pytest
import torch

import synth
from tests.test_gpu_attention import (_check_permuted_frontier, check_case,  # noqa: F401
                                      run_attention, ssd)

pytestmark = pytest.mark.gpu

SHORT, LONG = (16, [16, 21, 40, 46]), (900, [900, 907, 911, 925])


def case(name, heads, d, prefix, cache, seed=31, k_v=0):
    return synth.make_case(name, grid_h=10, grid_w=3 - 2 * k_v, prefix_len=prefix, cache_len=cache,
                           Hq=heads[0], Hkv=heads[1], d=d, V=64, seed=seed, k_v=k_v,
                           with_logits=False)


@pytest.mark.parametrize("heads", [(129, 1), (170, 1), (320, 2)])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("prefix,cache", [SHORT, LONG])
def test_matches_oracle(ssd, heads, d, prefix, cache):  # noqa: F811
    c = case("mma_sync", heads, d, prefix, cache)
    check_case(ssd, c)
    check_case(ssd, c, scale=0.05)


def test_the_most_heads(ssd):  # noqa: F811
    c = case("heads_256", (256, 1), 128, 500, [500, 503, 509], k_v=1)
    check_case(ssd, c)


@pytest.mark.parametrize("prefix,cache", [SHORT, LONG])
def test_shuffled_draft_order(ssd, prefix, cache):  # noqa: F811
    _check_permuted_frontier(ssd, case("mma_shuffled", (150, 1), 128, prefix, cache))


def test_split_merge_ignores_workspace_contents(ssd):  # noqa: F811
    """Partials in the workspace, merged by the combine kernel: whatever the workspace
    held before, the result is the same, bit for bit."""
    c, other = case("mma_ws", (150, 1), 128, *LONG), case("mma_ws2", (150, 1), 128, *LONG, seed=32)
    wsb = ssd.ssd_verify_attention_workspace(c.B, c.Hq, c.Hkv, c.d, c.D_max, c.L_max)
    assert wsb > 256  # split
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    outs = []
    for fill in (0xFF, 0x00, None, "other", None):
        if fill == "other":
            run_attention(ssd, other, ws=ws)
        elif fill is not None:
            ws.fill_(fill)
        outs.append(run_attention(ssd, c, ws=ws))
    for o, lse, _, st in outs:
        assert st == 0
        assert np.array_equal(o, outs[0][0]) and np.array_equal(lse, outs[0][1])


@pytest.mark.parametrize("prefix,cache", [SHORT, LONG])
def test_bad_draft_position_skips_only_its_sequence(ssd, prefix, cache):  # noqa: F811
    c = case("mma_bad", (150, 1), 128, prefix, cache)
    good = run_attention(ssd, c)

    def corrupt(pos):
        pos[1, 0] = c.grid_h * c.grid_w + 5

    o, _, _, st = run_attention(ssd, c, edit_pos=corrupt)
    assert good[3] == 0 and st == 6 and not o[1].any()
    rest = [b for b in range(c.B) if b != 1]
    assert np.array_equal(o[rest], good[0][rest])
