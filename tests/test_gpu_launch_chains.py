"""Library calls directly behind one another, with nothing between them, each reading
or overwriting what the one before read or wrote: every kernel that is launched as a
programmatic dependent must wait for what precedes it, so all buffers must end as
they do with a synchronisation after every call, bit for bit, launched and captured."""
import numpy as np
import pytest
import torch

from paper_2606_20543_gb300.step import VerifyStep
from tests.test_gpu_lmhead import ssd  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

B, W, H, PREFIX, HQ, HKV, D, V = 6, 64, 64, 256, 16, 8, 128, 4096
D_MAX, L_MAX = 2 * W, PREFIX + H * W


class Buffers:
    """Named device tensors with their first contents."""

    def __init__(self):
        self.g = torch.Generator(device="cuda").manual_seed(77)
        self.t, self.first = {}, {}

    def add(self, name, tensor):
        self.t[name] = tensor
        self.first[name] = tensor.clone()
        return tensor

    def normal(self, name, shape, dtype=torch.bfloat16, std=0.3):
        x = torch.randn(shape, device="cuda", generator=self.g) * std
        return self.add(name, x.to(dtype))

    def zeros(self, name, shape, dtype):
        return self.add(name, torch.zeros(shape, dtype=dtype, device="cuda"))

    def ints(self, name, values):
        return self.add(name, torch.tensor(values, dtype=torch.int32, device="cuda"))

    def reset(self):
        for k, t in self.t.items():
            t.copy_(self.first[k])
        torch.cuda.synchronize()

    def bits(self):
        torch.cuda.synchronize()
        return {k: t.cpu().contiguous().view(torch.uint8).numpy().copy() for k, t in self.t.items()}


def _check(b, calls):
    b.reset()
    for call in calls:
        call()
        torch.cuda.synchronize()
    want = b.bits()
    assert not any(want[k].any() for k in want if k.startswith("status"))
    for _ in range(3):
        b.reset()
        for call in calls:
            call()
        got = b.bits()
        assert [k for k in want if not np.array_equal(want[k], got[k])] == []
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for call in calls:
            call()
    for _ in range(3):
        b.reset()
        graph.replay()
        got = b.bits()
        assert [k for k in want if not np.array_equal(want[k], got[k])] == []


LENS = [PREFIX + n for n in (3900, 2000, 3001, 70, 3500, 1234)]
LENS2 = [PREFIX + n for n in (100, 3800, 64, 2500, 900, 3111)]


def _attention(lib, b, heads=(HQ, HKV), k_v=1):
    """Buffers of an attention over long caches and calls on them: (attention into o,
    attention into another o, frontier of a second set of lengths, in-place commit)."""
    Hq, Hkv = heads
    w = W if k_v else 3
    h = H if k_v else 1000
    d_max, l_max = (k_v + 1) * w, PREFIX + h * w
    grid = lib.grid(h, w, PREFIX, k_v=k_v)
    lens = [min(n, l_max - 1 - d_max) for n in LENS]
    lens2 = [min(n, l_max - 1 - d_max) for n in LENS2]
    cache, cache2 = b.ints("cache", lens), b.ints("cache2", lens2)
    n, pos = b.zeros("n", (B,), torch.int32), b.zeros("pos", (B, d_max), torch.int32)
    st = b.zeros("status", (1,), torch.int32)
    q, q2 = b.normal("q", (B, d_max, Hq, D)), b.normal("q2", (B, d_max, Hq, D))
    k, v = b.normal("k", (B, Hkv, l_max, D)), b.normal("v", (B, Hkv, l_max, D))
    o, o2 = (b.zeros(x, (B, d_max, Hq, D), torch.bfloat16) for x in ("o", "o2"))
    wsb = lib.ssd_verify_attention_workspace(B, Hq, Hkv, D, d_max, l_max)
    ws = torch.empty(max(wsb, 256), dtype=torch.uint8, device="cuda")

    def att(q, o):
        lib.ssd_verify_attention(grid, B, Hq, Hkv, D, cache, n, pos, d_max, l_max, q, k, v, 0.0,
                                 o, None, ws, wsb, st)

    def frontier(lengths):
        lib.ssd_frontier(grid, B, lengths, d_max, n, pos, st)

    frontier(cache)
    torch.cuda.synchronize()
    for x in ("n", "pos"):
        b.first[x].copy_(b.t[x])
    return dict(first=lambda: att(q, o), second=lambda: att(q2, o2), over=lambda: att(q2, o),
                frontier=lambda: frontier(cache), frontier2=lambda: frontier(cache2),
                commit=lambda: lib.ssd_commit_pass(grid, B, cache, d_max, "block", cache, st))


@pytest.mark.parametrize("heads,k_v", [((HQ, HKV), 1), ((150, 1), 0)])
@pytest.mark.parametrize("order", [
    ("first", "over"),                            # the same o written twice
    ("first", "commit", "frontier", "second"),    # cache, n_drafts and draft_pos overwritten
    ("first", "frontier", "second", "commit", "frontier"),
])
def test_attention_then_what_it_reads(ssd, order, heads, k_v):  # noqa: F811
    b = Buffers()
    c = _attention(ssd, b, heads, k_v)
    _check(b, [c[name] for name in order])


def _step_buffers(b, s, hidden=False):
    for name in ("q", "k", "v") + (("h_tgt", "h_drf") if hidden else ("tgt", "drf")):
        x = getattr(s, name)
        x.copy_(torch.randn(x.shape, device="cuda", generator=b.g) * (2.0 if name in ("tgt", "drf")
                                                                      else 0.3))
        b.add(name, x)
    if hidden:
        for x in (s.w_tgt, s.w_drf):
            x.copy_(torch.randn(x.shape, device="cuda", generator=b.g) * 0.05)
    s.cache_len.copy_(torch.tensor(LENS[:s.B], dtype=torch.int32))
    b.add("cache_len", s.cache_len)
    for name in ("o", "lse", "n_drafts", "draft_pos", "out_tok", "accepted", "ratio",
                 "accepted_count", "accepted_prefix", "next_cache_len"):
        getattr(s, name).zero_()
        b.add(name, getattr(s, name))
    b.add("status", s.status)


@pytest.mark.parametrize("strategy", ["accept_reject", "greedy"])
def test_attention_step_record_commit(ssd, strategy):  # noqa: F811
    """An attention on the step's own buffers, the step, the record of its tokens, the
    commit pass over its cache lengths in place, and the next step."""
    b = Buffers()
    s = VerifyStep(H, W, PREFIX, B, HQ, HKV, D, D_MAX, L_MAX, V, strategy=strategy)
    _step_buffers(b, s)
    s.set_rng(3, 1)
    s.track_grid()
    b.add("grid_tok", s.grid_tok)
    other = b.ints("other", LENS2)

    def front():
        ssd.ssd_frontier(s.g, B, other, D_MAX, s.n_drafts, s.draft_pos, s.status)

    def att():
        ssd.ssd_verify_attention(s.g, B, HQ, HKV, D, other, s.n_drafts, s.draft_pos, D_MAX, L_MAX,
                                 s.q, s.k, s.v, 0.0, s.o, s.lse, s.workspace, s.ws_bytes, s.status)

    def record():
        ssd.ssd_record_commit(B, D_MAX, PREFIX, H * W, s.cache_len, s.next_cache_len, s.out_tok,
                              s.grid_tok, s.status)

    def commit():
        ssd.ssd_commit_pass(s.g, B, s.cache_len, D_MAX, "first_row", s.cache_len, s.status)

    _check(b, [front, att, s.run, record, commit, s.run, record, front, att])


@pytest.mark.parametrize("images,V_,hidden", [(1, 2048, 256), (2, 4096, 512)])
def test_fused_steps_in_a_row(ssd, images, V_, hidden):  # noqa: F811
    """Fused steps of 128 rows (single CTAs) and 256 (pairs), and the fused acceptance
    alone, whose counts may overwrite the cache lengths."""
    b = Buffers()
    s = VerifyStep(H, W, PREFIX, images, HQ, HKV, D, D_MAX, L_MAX, V_, hidden=hidden)
    _step_buffers(b, s, hidden=True)
    s.set_rng(3, 1)

    def accept_in_place():
        keep = s.out.next_cache_len
        s.out.next_cache_len = s.cache_len.data_ptr()
        ssd.ssd_verify_accept(s.args, s.out, s.workspace, s.ws_bytes)
        s.out.next_cache_len = keep

    _check(b, [s.run, accept_in_place, s.run, accept_in_place])


def test_rounds_and_stage_shift(ssd):  # noqa: F811
    """Acceptance rounds, each on the tokens and references of the one before, with
    the trailing row moved to the front between them."""
    b = Buffers()
    rows, D2 = B * 2 * W, 2 * W
    tgts = [b.normal(f"tgt{i}", (rows, V), torch.float32, 2.0) for i in range(3)]
    drf = b.normal("drf", (rows, V), torch.float32, 2.0)
    refs = b.add("refs", ssd.row_addresses(drf))
    toks = [b.zeros(f"tok{i}", (rows,), torch.int32) for i in range(2)]
    acc, ratio = b.zeros("acc", (rows,), torch.uint8), b.zeros("ratio", (rows,), torch.float32)
    st = b.zeros("status", (1,), torch.int32)

    def one(i):
        def call():
            ssd.ssd_accept_round("accept_reject" if i != 1 else "sample", rows, V, tgts[i], V, refs,
                                 None if i == 0 else toks[(i + 1) % 2], 1.0, ssd.rng(5, i),
                                 toks[i % 2], acc, ratio, None, st)
        return call

    def plain():
        ssd.ssd_accept(rows, V, tgts[0], drf, V, None, 1.0, ssd.rng(5, 9), toks[1], acc, ratio,
                       None, st)

    _check(b, [one(0), one(1), lambda: ssd.ssd_stage_shift(B, D2, W, toks[1], refs), one(2), plain])


@pytest.mark.parametrize("rows", [24, 130])
def test_predictions_and_lm_heads(ssd, rows):  # noqa: F811
    """Draft predictions over one workspace, and lm_head acceptances whose draft tokens
    are the predictor's, then their own (130 rows: two predictor launches, CTA pairs)."""
    d, m, v_ = 512, 1024, 2048
    b = Buffers()
    z = [b.normal(f"z{i}", (rows, 2 * d), std=1.0) for i in range(2)]
    w0, w1, w3 = (b.normal(k, s, std=s[1] ** -0.5) for k, s in
                  (("w0", (d, 2 * d)), ("w1", (m, d)), ("w3", (m, d))))
    w2, wh = b.normal("w2", (d, m), std=m ** -0.5), b.normal("wh", (d, v_), std=d ** -0.5)
    g1, g2 = (b.normal(k, (d,), torch.float32, 1.0) for k in ("g1", "g2"))
    tok, hid = b.zeros("tok", (rows,), torch.int32), b.zeros("hid", (rows, d), torch.float32)
    st = b.zeros("status", (1,), torch.int32)
    wsb = ssd.ssd_draft_predict_workspace(rows, d, m, v_)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    hs = [b.normal(f"h{i}", (rows, d), std=1.0) for i in range(2)]
    out, acc = b.zeros("out", (rows,), torch.int32), b.zeros("acc", (rows,), torch.uint8)
    ratio = b.zeros("ratio", (rows,), torch.float32)
    lwsb = ssd.ssd_lmhead_accept_workspace(rows, v_)
    lws = torch.empty(lwsb, dtype=torch.uint8, device="cuda")

    def predict(i):
        return lambda: ssd.ssd_draft_predict(rows, d, m, v_, z[i], w0, w1, w3, w2, g1, g2, wh,
                                             1e-5, tok, hid, ws, wsb, st)

    def lm(i, drafts, result):
        return lambda: ssd.ssd_lmhead_accept(rows, v_, d, hs[i], hs[1 - i], wh, wh, drafts, 1.0,
                                             ssd.rng(7, i), result, acc, ratio, None, lws, lwsb, st)

    _check(b, [predict(0), lm(0, tok, out), predict(1), lm(1, out, tok), lm(0, tok, out),
               predict(0), predict(1)])
