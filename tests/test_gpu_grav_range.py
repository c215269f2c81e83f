"""The multigrid's integer neighbour sums over the exponent range: a solve is linear, so a
power of two on G scales every bit of the potential (values aligned by exponent, no absolute
threshold), also with a density contrast whose small potentials lie far below the largest;
and where everything is zero (the FP64 path) the potential is zero."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_37859_gb300 import workloads as wl  # noqa: E402
from test_gpu_hydro import Pair, tde, ctx  # noqa: E402,F401

pytestmark = pytest.mark.gpu


def phi(P, G, isolated):
    P.gm.gravity_solve(G, 0.0, tol=0.0, max_cycles=2, warm=False, isolated=isolated, fmg=True)
    return P.gm.gravity_phi().cpu().numpy().copy()


@pytest.mark.parametrize("isolated", [False, True])
@pytest.mark.parametrize("N", [(32, 32, 32), (16, 16, 8)])
def test_power_of_two_scales_the_potential(oracle, tde, ctx, N, isolated):
    h = max(N)
    lay = wl.uniform_layout(N, tuple(min(n, 16) for n in N), domain=tuple((-n / h, n / h) for n in N),
                            bc=(0, 0, 0) if isolated else (1, 1, 1), ng=2)
    rho = np.full((N[2], N[1], N[0]), 1e-12)
    rho[3, 5, 7] = 1.0
    z = 0 * rho
    P = Pair(oracle, tde, ctx, lay, wl.prim_state(lay, rho, z, z, z, 1 + z))
    a = phi(P, 1.0, isolated)
    assert np.isfinite(a).all() and np.abs(a).max() > 0
    for e in (-400, 400):
        assert np.array_equal(phi(P, 2.0 ** e, isolated), np.ldexp(a, e))


def test_uniform_periodic_density_has_no_potential(oracle, tde, ctx):
    lay = wl.uniform_layout((16, 16, 16), (16, 16, 16), bc=(1, 1, 1), ng=2)
    one = np.ones((16, 16, 16))
    P = Pair(oracle, tde, ctx, lay, wl.prim_state(lay, one, 0 * one, 0 * one, 0 * one, one))
    assert (phi(P, 1.0, False) == 0).all()
