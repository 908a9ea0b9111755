"""The draft predictor's sums run in one fixed order, and its tokens depend on it
where two logits nearly tie: tokens and hidden state against recorded bits, calls
in a row against each other, and tokens against 64-bit logits."""
import os
import zlib

import pytest
import torch

from tests.test_gpu_predictor import ssd  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "predictor_sums.txt")
SHAPES = [(24, 4096, 8192, 16384), (92, 896, 1792, 5120), (1, 512, 1024, 2048),
          (128, 1024, 2048, 4096)]
EPS = 1e-5
# A logit's error: bf16 roundings of the product inputs leave 1.5e-3 of the hidden
# state's norm and, in the rounded Hg, another 1.1e-3 (2^-9 / sqrt(3)), so 1.9e-3 of the
# logits' spread; the token's logit can be below the largest by the difference of
# two such errors, 5 standard deviations of which are 1.3e-2.
TIE = 1.5e-2


def _hash(shape, salt, scale):
    """Uniform values of standard deviation `scale` from integer arithmetic alone."""
    n = 1
    for k in shape:
        n *= k
    x = torch.arange(n, device="cuda", dtype=torch.int64).add_(salt * 40503).bitwise_and_(0xffffffff)
    x = x.mul_(747796405).add_(2891336453).bitwise_and_(0xffffffff)
    x.bitwise_xor_(x >> 16)
    x = x.mul_(277803737).bitwise_and_(0xffffffff)
    x.bitwise_xor_(x >> 15)
    return ((x >> 16).float() - 32767.5).mul_(scale * 3 ** 0.5 / 32768).view(shape)


def _weights(d, m, V, salt):
    w = {k: _hash(shape, salt + i, std).bfloat16() for i, (k, shape, std) in enumerate((
        ("w0", (d, 2 * d), (2 * d) ** -0.5), ("w1", (m, d), d ** -0.5), ("w3", (m, d), d ** -0.5),
        ("w2", (d, m), m ** -0.5), ("wh", (d, V), d ** -0.5)))}
    w["g1"], w["g2"] = 1 + _hash((d,), salt + 7, 0.1), 1 + _hash((d,), salt + 8, 0.1)
    return w


def _z(rows, d, salt):
    return _hash((rows, 2 * d), salt, 1.0).bfloat16()


def _calls(lib, w, z, V, n):
    """Tokens and hidden states of n calls in a row."""
    rows, d, m = z.shape[0], w["w0"].shape[0], w["w1"].shape[0]
    wsb = lib.ssd_draft_predict_workspace(rows, d, m, V)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    outs = [(torch.full((rows,), -7, dtype=torch.int32, device="cuda"),
             torch.zeros((rows, d), device="cuda")) for _ in range(n)]
    for tok, hid in outs:
        lib.ssd_draft_predict(rows, d, m, V, z, w["w0"], w["w1"], w["w3"], w["w2"], w["g1"],
                              w["g2"], w["wh"], EPS, tok, hid, ws, wsb, st)
    torch.cuda.synchronize()
    assert st.item() == 0
    return outs


def _record(lib, shape, salt):
    rows, d, m, V = shape
    (tok, hid), = _calls(lib, _weights(d, m, V, salt), _z(rows, d, salt + 9), V, 1)
    crc = zlib.crc32(hid.cpu().numpy().tobytes())
    return " ".join(str(int(x)) for x in (*shape, salt, crc, *tok.tolist()))


@pytest.mark.parametrize("shape", SHAPES)
def test_recorded_bits(ssd, shape):  # noqa: F811
    """The hidden state's checksum and the tokens as recorded on a GB300 (the order of
    the sums depends on the number of SMs).  A whole-K sum per tile instead of the
    partial sums in slot order changed 10 of 2304 tokens."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("recorded with 152 SMs")
    want = [line.strip() for line in open(GOLDEN) if line.startswith(" ".join(map(str, shape)))]
    assert len(want) >= 2
    for line in want:
        assert _record(ssd, shape, int(line.split()[4])) == line


@pytest.mark.parametrize("shape,weights,sets", [(SHAPES[0], 2, 8), (SHAPES[1], 2, 4),
                                                (SHAPES[3], 1, 4)])
def test_repeats_and_ties(ssd, shape, weights, sets):  # noqa: F811
    """Calls in a row on one workspace give the same bits, and every token that is not
    the 64-bit argmax belongs to a row whose logits tie within TIE."""
    rows, d, m, V = shape
    for i in range(weights):
        w = _weights(d, m, V, 100 * (i + 1))
        f = {k: w[k].double() for k in ("w0", "w1", "w3", "w2", "wh")}
        for s in range(sets):
            z = _z(rows, d, 100 * (i + 1) + 20 + s)
            outs = _calls(ssd, w, z, V, 4)
            for tok, hid in outs[1:]:
                assert torch.equal(tok, outs[0][0]) and torch.equal(hid, outs[0][1])
            a = z.double() @ f["w0"].T
            x = a / torch.sqrt((a * a).mean(1, keepdim=True) + EPS) * w["g1"].double()
            h = a + (torch.nn.functional.silu(x @ f["w1"].T) * (x @ f["w3"].T)) @ f["w2"].T
            assert (outs[0][1].double() - h).norm() < 2e-3 * h.norm()
            logits = (h * w["g2"].double()) @ f["wh"]
            short = logits.max(1).values - logits.gather(1, outs[0][0].long()[:, None])[:, 0]
            assert (short / logits.std(1)).max().item() < TIE
