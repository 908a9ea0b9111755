"""The calls this library is timed on: what a decoding program has it do.

A program that decodes images with spatial drafts calls, per backbone pass, the
draft predictor, the verification step (frontier, frontier attention,
acceptance, counts) or its fused-head form, and while it corrects a block, the
verify-and-correct rounds.  Engines that own their attention or their sampler
call the attention and the acceptance on their own.  Every case goes through
the package's public entry points on device buffers that such a program keeps.

Kinds of case:
  step     VerifyStep.run: one whole verification pass (logits path, or with
           `hidden` > 0 the fused lm_head path); `k_h` > 0 is the horizontal
           stage (k_h drafts along the row, bonus token)
  rounds   VerifyRounds.run: `rounds` verify-and-correct passes over one block
  attn     ssd_verify_attention alone
  accept   ssd_verify_accept: frontier, acceptance, committed draws, counts
  lmhead   ssd_lmhead_accept: hidden states and GenHead weights to decisions
  predict  ssd_draft_predict: Eq. 2's draft predictor and the draft tokens

Sizes are those of the repository's workloads (16x16, 24x24, 32x32 and 64x64
grids, 8 x 64 to 32 x 128 heads, vocabularies of 4096 to 65536, the 4096-wide
GenHead) and, in draw(), the ranges between them.
"""
import math

import torch

import paper_2606_20543_gb300 as ssd
from paper_2606_20543_gb300.step import VerifyRounds, VerifyStep

DEV = "cuda"


def _seq(lens):
    return ",".join(str(int(c)) for c in lens)


def listed():
    return [
        # smallest: one 16x16 image, 32 drafts, every kernel latency-bound
        dict(name="step_16x16_b1", kind="step", H=16, W=16, prefix=32, cache="192", Hq=8, Hkv=8,
             d=64, V=4096, k_v=1, k_h=0, hidden=0, logits="normal"),
        # one 24x24 image in the middle of its grid: the interactive, batch-1 call
        dict(name="step_24x24_b1", kind="step", H=24, W=24, prefix=120, cache="413", Hq=16, Hkv=16,
             d=128, V=16384, k_v=1, k_h=0, hidden=0, logits="normal"),
        # 24x24 images at every row of the grid in one ragged batch (one of them finished)
        dict(name="step_24x24_b25", kind="step", H=24, W=24, prefix=120,
             cache=_seq(range(120, 697, 24)), Hq=16, Hkv=16, d=128, V=16384, k_v=1, k_h=0,
             hidden=0, logits="normal"),
        # a served batch with grouped-query attention and uneven caches
        dict(name="step_32x32_gqa_b16", kind="step", H=32, W=32, prefix=64,
             cache="69,1030,511,257,866,142,733,388,950,604,201,1071,455,318,790,667", Hq=32,
             Hkv=8, d=128, V=16384, k_v=1, k_h=0, hidden=0, logits="zipf"),
        # the last passes of a 64x64 batch: one image left, the others complete
        dict(name="step_64x64_b8_tail", kind="step", H=64, W=64, prefix=256,
             cache="4352,4352,4170,4352,4352,4352,4352,4352", Hq=32, Hkv=32, d=128, V=65536,
             k_v=1, k_h=0, hidden=0, logits="zipf"),
        # the horizontal stage on the first row: five drafts and the bonus token
        dict(name="step_h5_24x24_b20", kind="step", H=24, W=24, prefix=120,
             cache=_seq(120 + i for i in range(20)), Hq=16, Hkv=16, d=128, V=16384, k_v=0, k_h=5,
             hidden=0, logits="normal"),
        # verify and correct: two rounds on the drafted rows, every rejected row redrawn
        dict(name="rounds2_24x24_b8", kind="rounds", H=24, W=24, prefix=120,
             cache="144,216,288,360,432,504,576,648", Hq=16, Hkv=16, d=128, V=16384, k_v=1,
             k_h=0, hidden=0, logits="normal", rounds=2),
        # the attention alone at long caches, 64x64 grids past their middle
        dict(name="attn_64x64_b8", kind="attn", H=64, W=64, prefix=256,
             cache="2300,2467,2711,2903,3125,3380,3555,3801", Hq=32, Hkv=32, d=128, k_v=1, k_h=0),
        # the acceptance alone at its largest: 1024 rows of a 65536 vocabulary
        dict(name="accept_64x64_b8", kind="accept", H=64, W=64, prefix=256,
             cache=_seq([256] * 8), V=65536, k_v=1, k_h=0, hidden=0, logits="zipf"),
        # the GenHead fused with the acceptance for one image's two drafted rows
        dict(name="lmhead_48", kind="lmhead", rows=48, V=16384, K=4096),
        # the fused step for five images: 240 rows through both GenHead products
        dict(name="step_fused_24x24_b5", kind="step", H=24, W=24, prefix=120,
             cache="120,240,360,480,600", Hq=16, Hkv=16, d=128, V=16384, k_v=1, k_h=0,
             hidden=4096, logits="normal"),
        # the draft predictor at the paper's head size, one 24-column grid row
        dict(name="predict_24", kind="predict", rows=24, d=4096, m=8192, V=16384),
    ]


def _log_int(rng, lo, hi, multiple=1):
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(x / multiple)) * multiple))


def _rand_grid(rng, B):
    W = rng.choice([16, 24, 32, 48, 64, rng.randrange(16, 64)])
    H = W
    prefix = rng.randrange(16, 257)
    # one image in ten is complete already (never the first)
    lens = [prefix + (H * W if b and rng.random() < 0.1 else rng.randrange(0, H * W))
            for b in range(B)]
    return H, W, prefix, lens


def draw(rng):
    kind = rng.choice(["step", "step", "step", "fused", "rounds", "attn", "attn", "accept",
                       "lmhead", "predict"])
    if kind == "predict":
        d = _log_int(rng, 512, 4096, 128)
        return dict(kind="predict", rows=rng.randrange(1, 129), d=d, m=2 * d,
                    V=_log_int(rng, 2048, 16384, 128))
    if kind == "lmhead":
        return dict(kind="lmhead", rows=_log_int(rng, 6, 256), V=_log_int(rng, 2048, 16384, 128),
                    K=_log_int(rng, 512, 4096, 64))
    if kind == "fused":
        B = rng.randrange(1, 6)
        H, W, prefix, lens = _rand_grid(rng, B)
        B = max(1, min(B, 256 // (2 * W)))
        return dict(kind="step", H=H, W=W, prefix=prefix, cache=_seq(lens[:B]), Hq=16, Hkv=16,
                    d=128, V=_log_int(rng, 2048, 16384, 128), k_v=1, k_h=0,
                    hidden=_log_int(rng, 512, 4096, 64), logits="normal")
    B = _log_int(rng, 1, 24)
    H, W, prefix, lens = _rand_grid(rng, B)
    Hq, Hkv, d = rng.choice([(8, 8, 64), (16, 16, 128), (32, 32, 128), (32, 8, 128), (12, 4, 64)])
    V = _log_int(rng, 4096, 65536, 4)
    horizontal = kind == "step" and rng.random() < 0.3
    k_v = 0 if horizontal else 1
    # at most what the largest listed cases hold: 1024 rows x 65536 entries, 64x64 caches of 8
    B = max(1, min(B, (1024 * 65536) // (2 * W * V), (8 * 32 * 4352) // (Hkv * (prefix + H * W))))
    case = dict(kind=kind, H=H, W=W, prefix=prefix, cache=_seq(lens[:B]), k_v=k_v,
                k_h=rng.randrange(3, 8) if horizontal else 0)
    if kind != "accept":
        case.update(Hq=Hq, Hkv=Hkv, d=d)
    if kind != "attn":
        case.update(V=V, hidden=0, logits=rng.choice(["normal", "zipf"]))
    if kind == "rounds":
        case.update(rounds=rng.randrange(2, 4))
        case["cache"] = _seq(lens[:max(1, B // 4)])
    largest = 1024 * 65536 * 8  # bytes of the largest listed case
    while work(case)["bytes"] > largest:
        case["cache"] = case["cache"].rpartition(",")[0]
    return case


# ------------------------------------------------------------------ the frontier
def _drafts(case):
    """Per sequence (cache length, drafts): the rest of the row (or its next
    k_h positions) and, when that completes the row, k_v rows below."""
    H, W, prefix = case["H"], case["W"], case["prefix"]
    out = []
    for text in case["cache"].split(","):
        c = int(text)
        y, x = divmod(c - prefix, W)
        n = 0
        if y < H:
            h = min(case["k_h"], W - x) if case["k_h"] else W - x
            n = h + (min(case["k_v"], H - 1 - y) * W if x + h == W else 0)
        out.append((c, n))
    return out


def _d_max(case):
    return (2 if case["k_h"] else case["k_v"] + 1) * case["W"]


def _l_max(case):
    return case["prefix"] + case["H"] * case["W"]


# ------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _normal(g, shape, std, dtype):
    return (torch.randn(shape, generator=g, device=DEV) * std).to(dtype)


def _fill_logits(g, tgt, drf, kind):
    """`normal`: N(0, 2^2) rows; `zipf`: draft logits -1.1 ln(rank) over a
    permutation of the vocabulary per row, target = draft + N(0, 2^2)."""
    rows, V = drf.shape
    if kind == "normal":
        drf.normal_(0.0, 2.0, generator=g)
        tgt.normal_(0.0, 2.0, generator=g)
        return
    base = -1.1 * torch.log(torch.arange(1, V + 1, device=DEV, dtype=torch.float32))
    for r0 in range(0, rows, 256):
        part = drf[r0:r0 + 256]
        perm = torch.rand(part.shape, generator=g, device=DEV).argsort(dim=1)
        part.copy_(base[perm])
    tgt.normal_(0.0, 2.0, generator=g).add_(drf)


def prepare(case, seed):
    g = _gen(seed)
    return {"step": _prepare_step, "rounds": _prepare_step, "accept": _prepare_step,
            "attn": _prepare_attn, "lmhead": _prepare_lmhead,
            "predict": _prepare_predict}[case["kind"]](case, g, seed)


def _prepare_step(case, g, seed):
    B = len(case["cache"].split(","))
    # the acceptance alone needs no attention buffers: the smallest legal ones
    Hq, Hkv, d = (case["Hq"], case["Hkv"], case["d"]) if "Hq" in case else (1, 1, 64)
    D_max = _d_max(case)
    s = VerifyStep(case["H"], case["W"], case["prefix"], B, Hq, Hkv, d, D_max, _l_max(case),
                   case["V"], hidden=case["hidden"], k_v=case["k_v"], k_h=case["k_h"], device=DEV,
                   commit="prefix_bonus" if case["k_h"] else "prefix")
    s.cache_len.copy_(torch.tensor([c for c, _ in _drafts(case)], dtype=torch.int32))
    for t in (s.q, s.k, s.v):
        t.copy_(_normal(g, t.shape, 0.125, torch.bfloat16))
    state = dict(kind=case["kind"], s=s)
    if case["hidden"]:
        for t, std in ((s.h_tgt, 1.0), (s.h_drf, 1.0), (s.w_tgt, 0.02), (s.w_drf, 0.02)):
            t.copy_(_normal(g, t.shape, std, torch.bfloat16))
    else:
        _fill_logits(g, s.tgt, s.drf, case["logits"])
    for t in (s.lse, s.out_tok, s.accepted, s.ratio):  # slots past the frontier stay as they are
        t.zero_()
    s.set_rng(seed, 0)
    if case["kind"] == "rounds":
        state["rounds"] = VerifyRounds(s)
        state["tgts"] = [s.tgt]
        for _ in range(case["rounds"] - 1):  # the backbone's rows drift from round to round
            t = state["tgts"][-1] * 0.6
            t.add_(torch.randn(t.shape, generator=g, device=DEV), alpha=0.8)
            state["tgts"].append(t)
        state["seed"] = seed
    return state


def _prepare_attn(case, g, seed):
    lens = _drafts(case)
    B, D_max, L_max = len(lens), _d_max(case), _l_max(case)
    Hq, Hkv, d = case["Hq"], case["Hkv"], case["d"]
    a = dict(kind="attn", B=B, Hq=Hq, Hkv=Hkv, d=d, D_max=D_max, L_max=L_max,
             grid=ssd.grid(case["H"], case["W"], case["prefix"], k_v=case["k_v"],
                           k_h=case["k_h"]))
    a["cache"] = torch.tensor([c for c, _ in lens], dtype=torch.int32, device=DEV)
    a["n"] = torch.empty(B, dtype=torch.int32, device=DEV)
    a["pos"] = torch.empty((B, D_max), dtype=torch.int32, device=DEV)
    a["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    ssd.ssd_frontier(a["grid"], B, a["cache"], D_max, a["n"], a["pos"], a["status"])
    a["q"] = _normal(g, (B, D_max, Hq, d), 0.125, torch.bfloat16)
    a["k"] = _normal(g, (B, Hkv, L_max, d), 0.125, torch.bfloat16)
    a["v"] = _normal(g, (B, Hkv, L_max, d), 0.125, torch.bfloat16)
    a["o"] = torch.zeros((B, D_max, Hq, d), dtype=torch.bfloat16, device=DEV)
    a["lse"] = torch.zeros((B, Hq, D_max), device=DEV)
    a["wsb"] = ssd.ssd_verify_attention_workspace(B, Hq, Hkv, d, D_max, L_max)
    a["ws"] = torch.empty(max(a["wsb"], 256), dtype=torch.uint8, device=DEV)
    return a


def _prepare_lmhead(case, g, seed):
    rows, V, K = case["rows"], case["V"], case["K"]
    a = dict(kind="lmhead", rows=rows, V=V, K=K, rng=ssd.rng(seed, 0))
    for name, shape, std in (("h_tgt", (rows, K), 1.0), ("h_drf", (rows, K), 1.0),
                             ("w_tgt", (K, V), 0.02), ("w_drf", (K, V), 0.02)):
        a[name] = _normal(g, shape, std, torch.bfloat16)
    a["out_tok"] = torch.zeros(rows, dtype=torch.int32, device=DEV)
    a["accepted"] = torch.zeros(rows, dtype=torch.uint8, device=DEV)
    a["ratio"] = torch.zeros(rows, device=DEV)
    a["lse"] = torch.zeros((rows, 2), device=DEV)
    a["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    a["wsb"] = ssd.ssd_lmhead_accept_workspace(rows, V)
    a["ws"] = torch.empty(a["wsb"], dtype=torch.uint8, device=DEV)
    return a


def _prepare_predict(case, g, seed):
    rows, d, m, V = case["rows"], case["d"], case["m"], case["V"]
    a = dict(kind="predict", rows=rows, d=d, m=m, V=V, eps=1e-5)
    for name, shape, std in (("z", (rows, 2 * d), 1.0), ("w0", (d, 2 * d), (2 * d) ** -0.5),
                             ("w1", (m, d), d ** -0.5), ("w3", (m, d), d ** -0.5),
                             ("w2", (d, m), m ** -0.5), ("w_head", (d, V), d ** -0.5)):
        a[name] = _normal(g, shape, std, torch.bfloat16)
    a["gamma1"] = 1.0 + 0.1 * torch.randn(d, generator=g, device=DEV)
    a["gamma2"] = 1.0 + 0.1 * torch.randn(d, generator=g, device=DEV)
    a["tok"] = torch.zeros(rows, dtype=torch.int32, device=DEV)
    a["hidden"] = torch.zeros((rows, d), device=DEV)
    a["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    a["wsb"] = ssd.ssd_draft_predict_workspace(rows, d, m, V)
    a["ws"] = torch.empty(a["wsb"], dtype=torch.uint8, device=DEV)
    return a


# --------------------------------------------------------------------------- run
def run(a):
    kind = a["kind"]
    if kind == "attn":
        ssd.ssd_verify_attention(a["grid"], a["B"], a["Hq"], a["Hkv"], a["d"], a["cache"], a["n"],
                                 a["pos"], a["D_max"], a["L_max"], a["q"], a["k"], a["v"], 0.0,
                                 a["o"], a["lse"], a["ws"], a["wsb"], a["status"])
        return dict(o=a["o"], lse=a["lse"], status=a["status"])
    if kind == "lmhead":
        ssd.ssd_lmhead_accept(a["rows"], a["V"], a["K"], a["h_tgt"], a["h_drf"], a["w_tgt"],
                              a["w_drf"], None, 1.0, a["rng"], a["out_tok"], a["accepted"],
                              a["ratio"], a["lse"], a["ws"], a["wsb"], a["status"])
        return {k: a[k] for k in ("out_tok", "accepted", "ratio", "lse", "status")}
    if kind == "predict":
        ssd.ssd_draft_predict(a["rows"], a["d"], a["m"], a["V"], a["z"], a["w0"], a["w1"],
                              a["w3"], a["w2"], a["gamma1"], a["gamma2"], a["w_head"], a["eps"],
                              a["tok"], a["hidden"], a["ws"], a["wsb"], a["status"])
        return dict(tok=a["tok"], hidden=a["hidden"], status=a["status"])
    s = a["s"]
    if kind == "rounds":
        r = a["rounds"]
        r.reset()
        r.run(a["tgts"], seed=a["seed"])
        # (the ratios of a later round belong to the tokens drawn before it)
        return dict(o=s.o, lse=s.lse, tokens=r.tokens, accepted=s.accepted,
                    accepted_count=s.accepted_count, accepted_prefix=s.accepted_prefix,
                    next_cache_len=s.next_cache_len, n_drafts=s.n_drafts, draft_pos=s.draft_pos,
                    status=s.status)
    if kind == "accept":
        ssd.ssd_verify_accept(s.args, s.out, s.workspace, s.ws_bytes)
    else:
        s.run()
    out = dict(out_tok=s.out_tok, accepted=s.accepted, ratio=s.ratio,
               accepted_count=s.accepted_count, accepted_prefix=s.accepted_prefix,
               next_cache_len=s.next_cache_len, n_drafts=s.n_drafts, draft_pos=s.draft_pos,
               status=s.status)
    if kind == "step":
        out.update(o=s.o, lse=s.lse)
    return out


# -------------------------------------------------------------------------- work
def work(case):
    """Each input read once, each output written once, of the part that the
    frontier needs: visible K/V once per KV head, Q and O of the drafts, both
    logit rows of every draft (or both GenHead matrices), the weights."""
    kind = case["kind"]
    if kind == "predict":
        rows, d, m, V = case["rows"], case["d"], case["m"], case["V"]
        w = 2 * d * d + 3 * d * m + d * V
        return dict(bytes=2 * w + rows * (4 * d + 4 * d + 4) + 8 * d, flops=2 * rows * w)
    if kind == "lmhead":
        rows, V, K = case["rows"], case["V"], case["K"]
        return dict(bytes=4 * K * V + 4 * rows * K + 17 * rows, flops=4 * rows * K * V)
    lens = _drafts(case)
    rounds = case.get("rounds", 1)
    nbytes = flops = 0
    for c, n in lens:
        if n == 0:
            continue
        if "Hq" in case:
            Hq, Hkv, d = case["Hq"], case["Hkv"], case["d"]
            nbytes += Hkv * (c + n) * d * 4 + n * Hq * (d * 4 + 4)
            flops += rounds * 4 * n * Hq * d * (c + n)
        rows = n + (1 if case["k_h"] else 0)
        if kind == "attn":
            continue
        if case["hidden"]:
            nbytes += rows * (4 * case["hidden"] + 9)
            flops += 4 * rows * case["hidden"] * case["V"]
        else:
            nbytes += rows * ((rounds + 1) * 4 * case["V"] + 9 * rounds)
            flops += rounds * 8 * rows * case["V"]
    if kind != "attn" and case["hidden"]:
        nbytes += 4 * case["hidden"] * case["V"]
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """About four times the error measured against 64 bits: 2e-3 for attention
    outputs (P and O are rounded to bf16), 1.2e-5 for the ratios of the fused
    GenHead (logits accumulated in fp32 over K = 4096), 1.5e-3 for the
    predictor (bf16 product inputs between the products), up to 8e-7 for the
    ratios of fp32 logits.  `differ`: decisions and draws at a tie."""
    kind = case["kind"]
    if kind == "accept":
        return dict(rel=1e-5, max=1e-4, differ=0.01)
    if kind == "lmhead":
        return dict(rel=6e-5, max=6e-4, differ=0.01)
    if kind == "predict":
        return dict(rel=6e-3, max=0.06, differ=0.01)
    return dict(rel=1e-2, max=0.1, differ=0.01)


# ------------------------------------------------------------------------- exact
def _exact_attention(case, q, k, v):
    B, D_max, Hq, d = q.shape
    G = Hq // case["Hkv"]
    o = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    lse = torch.zeros((B, Hq, D_max), dtype=torch.float64, device=DEV)
    for b, (c, n) in enumerate(_drafts(case)):
        if n == 0:
            continue
        qb = q[b, :n].double().transpose(0, 1)                               # [Hq, n, d]
        kb = k[b, :, :c + n].double().repeat_interleave(G, dim=0)            # [Hq, c + n, d]
        vb = v[b, :, :c + n].double().repeat_interleave(G, dim=0)
        s = qb @ kb.transpose(1, 2) / math.sqrt(d)
        key = torch.arange(c + n, device=DEV)
        s.masked_fill_(key[None, :] > (c + torch.arange(n, device=DEV))[:, None], -math.inf)
        lse[b, :, :n] = torch.logsumexp(s, dim=2)
        o[b, :n] = (torch.softmax(s, dim=2) @ vb).transpose(0, 1)
    return o, lse


def _exact_ratio(tgt, drf):
    """Ratio p(t) / q(t) at t = argmax q and both log-sum-exps, in 64 bits."""
    tgt, drf = tgt.double(), drf.double()
    lse = torch.stack([torch.logsumexp(tgt, 1), torch.logsumexp(drf, 1)], 1)
    t = drf.argmax(dim=1, keepdim=True)
    ratio = torch.exp((tgt.gather(1, t) - drf.gather(1, t)).squeeze(1) - lse[:, 0] + lse[:, 1])
    return ratio, lse


def _exact_rows(a, rows):
    s = a["s"]
    if s.tgt is not None:
        return _exact_ratio(s.tgt[rows], s.drf[rows])[0]
    return _exact_ratio(s.h_tgt[rows].double() @ s.w_tgt.double(),
                        s.h_drf[rows].double() @ s.w_drf.double())[0]


def exact(case, seed):
    a = prepare(case, seed)
    kind = case["kind"]
    if kind == "attn":
        o, lse = _exact_attention(case, a["q"], a["k"], a["v"])
        return dict(o=o, lse=lse, status=None)
    if kind == "lmhead":
        ratio, lse = _exact_ratio(a["h_tgt"].double() @ a["w_tgt"].double(),
                                  a["h_drf"].double() @ a["w_drf"].double())
        return dict(out_tok=None, accepted=None, ratio=ratio, lse=lse, status=None)
    if kind == "predict":
        f = {k: a[k].double() for k in ("z", "w0", "w1", "w3", "w2")}
        A = f["z"] @ f["w0"].T
        x = A / torch.sqrt((A * A).mean(1, keepdim=True) + a["eps"]) * a["gamma1"].double()
        h = A + (torch.nn.functional.silu(x @ f["w1"].T) * (x @ f["w3"].T)) @ f["w2"].T
        return dict(tok=None, hidden=h, status=None)
    s = a["s"]
    names = ("accepted", "accepted_count", "accepted_prefix", "next_cache_len", "n_drafts",
             "draft_pos", "status")
    out = dict.fromkeys(names)
    if kind == "rounds":
        out["tokens"] = None
    else:
        out["out_tok"] = None
        ratio = torch.zeros(s.rows, dtype=torch.float64, device=DEV)
        for b, (_, n) in enumerate(_drafts(case)):
            if n:
                rows = slice(b * s.D_max, b * s.D_max + n)
                ratio[rows] = _exact_rows(a, rows)
        out["ratio"] = ratio
    if kind != "accept":
        out["o"], out["lse"] = _exact_attention(case, s.q, s.k, s.v)
    return out
