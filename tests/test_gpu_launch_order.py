"""Calls in a row on one stream, each after copies that overwrite its inputs (by
a kernel, or on a second stream joined by an event) and before a copy of its
outputs: every kernel is launched as a programmatic dependent of what precedes
it, so the results must be those of calls with a synchronisation between, bit
for bit, launched and captured."""
import numpy as np
import pytest
import torch

from paper_2606_20543_gb300.step import VerifyStep
from tests.test_gpu_lmhead import ssd  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

D, B, V = 64, 3, 4096


def _inputs(s, seed):
    """Values for the inputs of the VerifyStep `s`."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    hw = s.g.grid_h * s.g.grid_w
    names = ["q", "k", "v"] + (["h_tgt", "h_drf"] if s.hidden else ["tgt", "drf"])
    x = {k: torch.randn(getattr(s, k).shape, device="cuda", generator=g).to(getattr(s, k).dtype)
         for k in names}
    x["cache_len"] = torch.tensor([s.g.prefix_len + n for n in (seed, 3 * seed, hw // 2)],
                                  dtype=torch.int32, device="cuda")
    return x


OUT = ("o", "n_drafts", "draft_pos", "out_tok", "accepted", "ratio", "accepted_count",
       "accepted_prefix", "next_cache_len")


@pytest.mark.parametrize("joined", [False, True])
@pytest.mark.parametrize("side,k_v,hidden,strategy,Hq,Hkv", [
    (8, 1, 0, "accept_reject", 4, 4),    # acceptance, attention, counts and draws
    (8, 1, 0, "greedy", 4, 2),           # counts without draws
    (8, 1, 128, "accept_reject", 4, 4),  # frontier, lm_head, attention, counts
    (3, 0, 0, "accept_reject", 129, 1),  # above 128 heads per KV head: a second stream
])
def test_calls_in_a_row(ssd, side, k_v, hidden, strategy, Hq, Hkv, joined):  # noqa: F811
    D_max, prefix = (k_v + 1) * side, 16
    s = VerifyStep(4 * side, side, prefix, B, Hq, Hkv, D, D_max, prefix + 4 * side * side, V,
                   hidden=hidden, strategy=strategy, k_v=k_v)
    if hidden:
        g = torch.Generator(device="cuda").manual_seed(9)
        for w in (s.w_tgt, s.w_drf):
            w.copy_(torch.randn(w.shape, device="cuda", generator=g) * 0.1)
    s.upload(cache_len=np.full(B, prefix, np.int32),
             uniforms=np.random.default_rng(5).random((s.rows, 2), np.float32))
    sets = [_inputs(s, seed) for seed in (1, 2, 3, 4)]
    for k, v in sets[0].items():
        getattr(s, k).copy_(v)
    outs = [{k: torch.zeros_like(getattr(s, k)) for k in OUT} for _ in sets]
    other = torch.cuda.Stream()

    def chain(sync):
        for x, y in zip(sets, outs):
            if joined:  # the inputs arrive on another stream
                cur = torch.cuda.current_stream()
                other.wait_stream(cur)
                with torch.cuda.stream(other):
                    for k, v in x.items():
                        getattr(s, k).copy_(v)
                cur.wait_stream(other)
            else:
                for k, v in x.items():
                    torch.add(v, 0, out=getattr(s, k))  # a kernel
            if sync:
                torch.cuda.synchronize()
            s.run()
            if sync:
                torch.cuda.synchronize()
            for k in OUT:
                y[k].copy_(getattr(s, k))

    def bits():
        torch.cuda.synchronize()
        r = [{k: v.cpu().contiguous().view(torch.uint8).numpy().copy() for k, v in y.items()}
             for y in outs]
        for y in outs:
            for v in y.values():
                v.zero_()
        return r

    s.run()
    torch.cuda.synchronize()
    s.o.zero_()
    chain(sync=True)
    want = bits()
    for _ in range(3):
        s.o.zero_()
        chain(sync=False)
        got = bits()
        assert all(np.array_equal(a[k], b[k]) for a, b in zip(want, got) for k in OUT)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(sync=False)
    for _ in range(3):
        s.o.zero_()
        graph.replay()
        got = bits()
        assert all(np.array_equal(a[k], b[k]) for a, b in zip(want, got) for k in OUT)
    assert not s.status.any()
