"""The full-multigrid start on grids whose large levels have no prolongation tiles (flat
grids, thin boxes): a lane per cell inside, a warp per cell along isolated faces, with the
line between the two forms crossed on the way up."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_37859_gb300 import workloads as wl  # noqa: E402
from test_gpu_grav import G, oracle_phi_iso  # noqa: E402,F401
from test_gpu_hydro import Pair, tde, ctx  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [(256, 256, 1), (64, 2048, 1), (256, 128, 4), (128, 256, 2)])
def test_isolated_fmg_matches_oracle(oracle, tde, ctx, N):
    h = max(N)
    lay = wl.uniform_layout(N, tuple(min(n, 32) for n in N), domain=tuple((-n / h, n / h) for n in N), bc=(0, 0, 0), ng=2)
    P = Pair(oracle, tde, ctx, lay, wl.random_smooth(lay, seed=3, drho=0.4, P0=1.0))
    P.gm.gravity_solve(G, 0.0, tol=0.0, max_cycles=1, warm=False, isolated=True, fmg=True)
    got = P.gm.gravity_phi().cpu().numpy()
    want = oracle_phi_iso(oracle, P, 1, True)[0]
    # the same cycles in another order of roundings (the bound of the other gravity tests)
    assert np.allclose(got, want, rtol=0, atol=1e-12 * np.abs(want).max())


@pytest.mark.parametrize("N", [(512, 512, 1), (256, 64, 4)])
def test_periodic_fmg_converges(oracle, tde, ctx, N):
    lay = wl.uniform_layout(N, tuple(min(n, 32) for n in N), domain=tuple((0, n / max(N)) for n in N), bc=(1, 1, 1), ng=2)
    P = Pair(oracle, tde, ctx, lay, wl.random_smooth(lay, seed=5, drho=0.4, P0=1.0))
    _, start = P.gm.gravity_solve(G, 0.0, tol=0.0, max_cycles=0, warm=False, fmg=False)
    _, fmg = P.gm.gravity_solve(G, 0.0, tol=0.0, max_cycles=0, warm=False, fmg=True)
    assert np.isfinite(fmg) and fmg < 0.1 * start   # (a cycle alone reduces it tenfold)
    n, d = P.gm.gravity_solve(G, 0.0, tol=1e-11, max_cycles=30, warm=False, fmg=True)
    m, e = P.gm.gravity_solve(G, 0.0, tol=1e-11, max_cycles=30, warm=False, fmg=False)
    assert d < 1e-11 and e < 1e-11 and n <= m
