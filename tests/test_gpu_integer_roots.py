"""The integer reciprocal, sqrt(a / b) and 1/sqrt(t) of the hydro kernels over the
whole exponent range and at the ends of a binade (powers of two and their
neighbours), where their normalisation and rounding carry can go wrong."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["powers", "below", "above", "random"])
def test_within_one_ulp_over_all_exponents(which):
    from paper_2609_37859_gb300 import tde
    ctx = tde.Context(0)
    k = np.arange(-1021, 1021)
    x = np.ldexp(1.0, k)
    rng = np.random.default_rng(5)
    if which == "below":
        x = np.nextafter(x, 0.0)[1:]
    elif which == "above":
        x = np.nextafter(x, np.inf)
    elif which == "random":
        x = np.ldexp(1.0 + rng.random(k.size), k)
    y = rng.permutation(x)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    out = torch.empty_like(xd)

    def probe(op, a, b=None):
        ctx.math_probe(op, a, out, b)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    # the forms are within 0.52 ulp of the exact value: at most one ulp from the
    # correctly rounded one (in extended precision where numpy has it)
    X, Y = x.astype(np.longdouble), y.astype(np.longdouble)
    for got, want in ((probe(tde.MATH_RCP, xd), 1 / X), (probe(tde.MATH_RCP, -xd), -1 / X),
                      (probe(tde.MATH_SQRT_RATIO, xd, yd), np.sqrt(X) / np.sqrt(Y)),
                      (probe(tde.MATH_RSQRT, xd), 1 / np.sqrt(X))):
        w = want.astype(np.float64)
        assert np.max(np.abs(got - w) / np.spacing(np.abs(w))) <= 1.0
