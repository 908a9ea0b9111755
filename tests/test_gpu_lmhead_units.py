"""The fused lm_head at the sizes where its ring units change shape, against
the oracle, and the fused step, whose attention runs on the SMs that the
lm_head leaves, against its parts, bit for bit, launched and captured."""
import numpy as np
import pytest
import torch

from oracle import lmhead as olm
from tests.helpers import FUSED_PROB_TOL, bf16_to_f64, compare_decisions, max_excused_rows
from tests.test_gpu_lmhead import make_inputs, run_fused, ssd  # noqa: F401 (ssd: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,K,V", [
    (1, 64, 128),      # one unit of 64 K, one CTA, one staged group of 8 rows
    (41, 192, 384),    # K not a multiple of 128: units of 64; a ragged row group, three CTAs
    (88, 384, 512),    # the most rows of 128-K units, an odd number of them
    (128, 384, 512),   # the most rows of one CTA
    (129, 384, 512),   # the fewest on CTA pairs
    (256, 128, 640),   # the most rows; five tiles, the third pair half empty
    # the search: 70 tiles (half a warp per row, 8 tiles per lane, one load each), 133
    # and 148 tiles (a warp per row; 148 in 16-byte loads), more rows than one pass takes
    (90, 64, 8960), (40, 64, 17024), (90, 64, 18944),
    # the most tiles, one per SM: single CTAs, pairs, and pairs of an odd number of tiles
    (8, 64, 19456), (160, 64, 19456), (200, 128, 19328),
])
def test_unit_shapes_match_oracle(ssd, rows, K, V):  # noqa: F811
    ht, hd, wt, wd, u = make_inputs(rows, K, V, 60 + rows, 0.1)
    tok, acc, ratio, lse, st = run_fused(ssd, ht, hd, wt, wd, u)
    assert st == 0
    ref = olm.lmhead_accept(bf16_to_f64(ht), bf16_to_f64(hd), bf16_to_f64(wt), bf16_to_f64(wd), u)
    assert compare_decisions(ref, tok, acc, ratio, lse, what=f"rows={rows} V={V}",
                             tol=FUSED_PROB_TOL) <= max_excused_rows(rows)


@pytest.mark.parametrize("rows", [8, 160])
def test_more_tiles_than_resident_ctas_are_refused(ssd, rows):  # noqa: F811
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ht, hd, wt, wd, u = make_inputs(rows, 64, 128 * (sms + 1), 5, 0.1)
    with pytest.raises(ssd.SsdError) as e:
        run_fused(ssd, ht, hd, wt, wd, u)
    assert e.value.code == 3  # SSD_ERR_UNSUPPORTED


@pytest.mark.parametrize("side,lens,V,hidden", [
    (8, [16, 40, 80], 128, 64),             # one lm_head CTA: the attention fits beside it
    (24, [120, 400, 696], 18944, 256),      # 148 CTAs: 4 of 152 SMs left
    (64, [4300, 4200], 2048, 512),          # a long attention beside 16 CTAs
])
def test_fused_step_is_its_parts(ssd, side, lens, V, hidden):  # noqa: F811
    from paper_2606_20543_gb300.step import VerifyStep
    prefix = {8: 16, 24: 120, 64: 256}[side]
    B, D_max, L_max = len(lens), 2 * side, prefix + side * side
    s = VerifyStep(side, side, prefix, B, 4, 4, 128, D_max, L_max, V, hidden=hidden)
    rng = np.random.default_rng(V)
    g = torch.Generator(device="cuda").manual_seed(V)
    bf = lambda *shape, std=1.0: (  # noqa: E731
        torch.randn(shape, device="cuda", generator=g) * std).bfloat16()
    s.upload(cache_len=np.array(lens, np.int32), q=bf(B, D_max, 4, 128), k=bf(B, 4, L_max, 128),
             v=bf(B, 4, L_max, 128), h_tgt=bf(B * D_max, hidden), h_drf=bf(B * D_max, hidden),
             w_tgt=bf(hidden, V, std=0.05), w_drf=bf(hidden, V, std=0.05),
             uniforms=rng.random((B * D_max, 2), np.float32))

    def bits(r):
        return {k: np.ascontiguousarray(v).view(np.uint8) for k, v in r.items()}

    def wipe():
        for t in (s.o, s.lse, s.out_tok, s.accepted, s.ratio, s.accepted_count, s.accepted_prefix,
                  s.next_cache_len, s.n_drafts, s.draft_pos):
            t.fill_(3)

    wipe()
    s.run()
    torch.cuda.synchronize()
    first = bits(s.results())
    assert not s.results()["status"].any()
    wipe()
    ssd.ssd_verify_accept(s.args, s.out, s.workspace, s.ws_bytes)
    ssd.ssd_verify_attention(s.g, B, 4, 4, 128, s.cache_len, s.n_drafts, s.draft_pos, D_max, L_max,
                             s.q, s.k, s.v, 0.0, s.o, s.lse, s.workspace, s.ws_bytes, s.status)
    torch.cuda.synchronize()
    parts = bits(s.results())
    wipe()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.run()
    graph.replay()
    torch.cuda.synchronize()
    replayed = bits(s.results())
    for k in first:
        assert np.array_equal(first[k], parts[k]), k
        assert np.array_equal(first[k], replayed[k]), k


def test_pair_gives_up_and_the_context_stays_usable(ssd):  # noqa: F811
    """CTA pairs leave together when a grid barrier runs out."""
    rows, K, V = 160, 256, 1024
    ht, hd, wt, wd, u = make_inputs(rows, K, V, 23, 0.05)
    ssd.ssd_set_wait_limit(1 << 12)
    ssd.ssd_set_barrier_shortfall(1)
    try:
        tok, acc, _, _, st = run_fused(ssd, ht, hd, wt, wd, u)
    finally:
        ssd.ssd_set_barrier_shortfall(0)
        ssd.ssd_set_wait_limit(0)
    assert st == 5 and np.all(tok == -7) and np.all(acc == 7)  # SSD_ERR_TIMEOUT, nothing written
    tok, acc, ratio, lse, st = run_fused(ssd, ht, hd, wt, wd, u)
    assert st == 0
    ref = olm.lmhead_accept(bf16_to_f64(ht), bf16_to_f64(hd), bf16_to_f64(wt), bf16_to_f64(wd), u)
    compare_decisions(ref, tok, acc, ratio, lse, what="pair after a timeout", tol=FUSED_PROB_TOL)
