"""A step whose Q or O is aligned to 4 or 8 bytes only (views into larger buffers): the
attention runs without TMA loads of Q and 16-byte stores of O, launched and
captured, and everything else is as with aligned buffers, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2606_20543_gb300.step import VerifyStep
from tests.helpers import ATTN_TOL, attention_error
from tests.test_gpu_lmhead import ssd  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q_off,o_off", [(2, 0), (0, 2), (4, 4)])
@pytest.mark.parametrize("Hq,Hkv,d,hidden", [(12, 4, 64, 0), (4, 4, 128, 0), (4, 4, 128, 128)])
def test_unaligned_q_and_o(ssd, Hq, Hkv, d, hidden, q_off, o_off):  # noqa: F811
    side, prefix, B, V = 12, 20, 3, 1024
    s = VerifyStep(side, side, prefix, B, Hq, Hkv, d, 2 * side, prefix + side * side, V,
                   hidden=hidden)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = {k: torch.randn(getattr(s, k).shape, device="cuda", generator=g) * 0.3
         for k in ("q", "k", "v") + (("h_tgt", "h_drf", "w_tgt", "w_drf") if hidden
                                     else ("tgt", "drf"))}
    s.upload(cache_len=np.array([prefix, prefix + 50, prefix + 131], np.int32),
             uniforms=np.random.default_rng(4).random((s.rows, 2), np.float32))
    for k, v in x.items():
        getattr(s, k).copy_(v)
    s.run()
    torch.cuda.synchronize()
    want = s.results()
    assert not want["status"].any()

    def view(t, off):
        big = torch.zeros(t.numel() + 16, dtype=t.dtype, device="cuda")
        assert big.data_ptr() % 16 == 0
        return big[off:off + t.numel()].view(t.shape)

    q, o = view(s.q, q_off), view(s.o, o_off)
    q.copy_(s.q)
    s.args.q, s.out.o, s.o = q.data_ptr(), o.data_ptr(), o
    for launch in ("call", "graph"):
        for t in (o, s.out_tok, s.accepted, s.next_cache_len):
            t.zero_()
        if launch == "call":
            s.run()
        else:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                s.run()
            graph.replay()
        torch.cuda.synchronize()
        got = s.results()
        for k in want:
            if k not in ("o", "lse"):
                assert np.array_equal(want[k], got[k]), (launch, k)
        for b in range(B):
            n = int(want["n_drafts"][b])
            assert n > 0 and np.abs(got["lse"][b, :, :n] - want["lse"][b, :, :n]).max() < 2e-2
            for h in range(Hq):
                assert attention_error(got["o"][b, :n, h], want["o"][b, :n, h]) < ATTN_TOL
