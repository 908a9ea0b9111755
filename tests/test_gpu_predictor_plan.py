"""The draft predictor at the sizes where its tile plan changes shape, against
the oracle (tokens exact but for argmax near-ties, hidden state within 2e-3)."""
import pytest

from tests.test_gpu_predictor import _case, _check, _run, ssd  # noqa: F401 (ssd: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,d,m,V", [
    (64, 384, 640, 1152),    # the most rows of M = 64 products; a last unit of part of the K
    (65, 384, 640, 1152),    # the fewest of M = 128
    (7, 2432, 256, 640),     # a last tile of 128 of the 2432 features (tiles of 16 on <= 152 SMs)
    (3, 128, 10240, 256),    # more gate tiles than CTAs: two rounds of one phase
    (24, 128, 256, 20480),   # more GenHead tiles than CTAs, 128 wide
    (40, 256, 384, 9856),    # 64-wide GenHead tiles against 128-wide ones
])
def test_predictor_plan_shapes(ssd, rows, d, m, V):  # noqa: F811
    w, g1, g2 = _case(170 + rows, rows, d, m, V)
    tok, hid = _run(ssd, rows, d, m, V, w, g1, g2, 1e-6)
    assert _check(w, g1, g2, 1e-6, tok, hid) <= max(1, rows // 10)
