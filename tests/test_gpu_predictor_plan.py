"""The draft predictor at the sizes where its tile plan changes shape, against
the oracle (tokens exact but for argmax near-ties, hidden state within 2e-3)."""
import pytest

from tests.test_gpu_predictor import _case, _check, _run, ssd  # noqa: F401 (ssd: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,d,m,V", [
    (64, 384, 640, 1152),    # four groups of 16 rows on N, and the first row of a fifth: two
    (65, 384, 640, 1152),    # tensor-memory column blocks and three
    (7, 2432, 256, 640),     # tiles of 38 units shared by 8 CTAs, which bounds the CTA count
    (3, 128, 10240, 256),    # two CTAs (a phase of two units) for 80 gate tiles
    (24, 128, 256, 20480),   # and for 160 GenHead tiles
    (40, 256, 384, 9856),    # 77 GenHead tiles on 6 CTAs, whose ranges cut tiles
])
def test_predictor_plan_shapes(ssd, rows, d, m, V):  # noqa: F811
    w, g1, g2 = _case(170 + rows, rows, d, m, V)
    tok, hid = _run(ssd, rows, d, m, V, w, g1, g2, 1e-6)
    assert _check(w, g1, g2, 1e-6, tok, hid) <= max(1, rows // 10)
