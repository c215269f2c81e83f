"""The stated error bounds of the integer reciprocal (0.51 ulp), sqrt(a / b) and 1/sqrt(t)
(0.52 ulp) against extended precision, over random significands of both exponent parities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ea,eb", [(0, 0), (1, 0), (0, 1), (301, -200)])
def test_bounds(ea, eb):
    from paper_2609_37859_gb300 import tde
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision")
    ctx = tde.Context(0)
    rng = np.random.default_rng(11)
    n = 1 << 19
    x, y = np.ldexp(1 + rng.random(n), ea), np.ldexp(1 + rng.random(n), eb)
    X, Y = x.astype(np.longdouble), y.astype(np.longdouble)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    out = torch.empty_like(xd)
    for op, b, want, bound in ((tde.MATH_RCP, None, 1 / X, 0.51), (tde.MATH_SQRT_RATIO, yd, np.sqrt(X / Y), 0.52),
                               (tde.MATH_RSQRT, None, 1 / np.sqrt(X), 0.52)):
        ctx.math_probe(op, xd, out, b)
        got = out.cpu().numpy().astype(np.longdouble)
        assert np.max(np.abs(got - want) / np.spacing(want.astype(np.float64))) <= bound
