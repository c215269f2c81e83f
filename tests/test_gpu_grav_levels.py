"""Multigrid V-cycles on grids that take each form of the level kernels: cubic and
flat cells, levels halved in some directions only, 16^3 and 8^3 prolongation
tiles and the untiled form, and grids that go into the one-CTA coarse cycle
whole or from some level down."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_37859_gb300 import workloads as wl  # noqa: E402
from test_gpu_grav import G, oracle_phi, oracle_phi_iso  # noqa: E402,F401
from test_gpu_hydro import Pair, tde, ctx  # noqa: E402,F401

pytestmark = pytest.mark.gpu

CUBIC = [(128, 128, 128), (64, 32, 16), (32, 32, 32), (16, 16, 8), (8, 8, 8), (4, 2, 2)]
FLAT = [(32, 16, 8), (16, 16, 64), (32, 64, 1), (8, 4, 4), (16, 1, 1)]


@pytest.mark.parametrize("form", ["periodic", "isolated", "isolated_fmg"])
@pytest.mark.parametrize("N,cubic", [(n, True) for n in CUBIC] + [(n, False) for n in FLAT])
def test_cycles_match_oracle(oracle, tde, ctx, N, cubic, form):
    isolated, fmg = form != "periodic", form == "isolated_fmg"
    h = max(N)
    dom = tuple((-n / h, n / h) for n in N) if cubic else ((-1, 1), (-0.7, 0.7), (-0.4, 0.4))
    block = tuple(min(n, 32) for n in N)
    bc = (0, 0, 0) if isolated else (1, 1, 1)
    lay = wl.uniform_layout(N, block, domain=dom, bc=bc, ng=2)
    W = wl.random_smooth(lay, seed=3, drho=0.4, P0=1.0)
    P = Pair(oracle, tde, ctx, lay, W)
    P.gm.gravity_solve(G, 0.0, tol=0.0, max_cycles=2, warm=False, isolated=isolated, fmg=fmg)
    got = P.gm.gravity_phi().cpu().numpy()
    want = oracle_phi_iso(oracle, P, 2, fmg)[0] if isolated else oracle_phi(oracle, P, P.U, 2)[0]
    # the same cycles in another order of roundings (the bound of the other gravity tests)
    assert np.allclose(got, want, rtol=0, atol=1e-12 * np.abs(want).max())
