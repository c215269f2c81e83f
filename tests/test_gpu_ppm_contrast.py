"""A PPM interface never leaves the interval between its two cells: steep drops onto a floor
more than 2^53 below, beside a step, where the fourth-order value lands on twice the drop
exactly (7, 1, floor).  The face densities and pressures stay positive, so a step stays
finite, as the oracle's does.  (Cell by cell the two differ: the fourth-order value cancels
there to rounding errors of the high side, which exceed the floor.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_37859_gb300 import workloads as wl  # noqa: E402
from test_gpu_hydro import Pair, tde, ctx  # noqa: E402,F401

pytestmark = pytest.mark.gpu

DROPS = [(7.0, 1.0, 1e-20), (49.0, 7.0, 1e-17), (7e-3, 1e-3, 1e-20), (1.0, 0.5, 1e-18)]


@pytest.mark.parametrize("drop", DROPS)
@pytest.mark.parametrize("riemann", [0, 1])
@pytest.mark.parametrize("axis,rising", [(0, False), (1, True), (2, False)])
@pytest.mark.parametrize("pressure", ["uniform", "density"])
def test_step_beside_a_floor(oracle, tde, ctx, drop, riemann, axis, rising, pressure):
    n = 16
    lay = wl.uniform_layout((n,) * 3, (n,) * 3, bc=(0, 0, 0), ng=3)
    line = np.full(n, drop[2])
    line[:7], line[7] = drop[0], drop[1]
    if rising:
        line = line[::-1]
    shape = [1, 1, 1]
    shape[2 - axis] = n
    rho = np.broadcast_to(line.reshape(shape), (n, n, n)).copy()
    z = 0 * rho
    W = wl.prim_state(lay, rho, z, z, z, rho if pressure == "density" else z + 1.0)
    P = Pair(oracle, tde, ctx, lay, W, recon=1, riemann=riemann, rho_floor=1e-25, p_floor=1e-25)
    U = P.U.copy()
    d = P.om.cfl_dt(U, 0.3).min()
    P.om.step(U, d, 0.0)
    P.gm.step(cfl=0.3)
    got, want = lay.to_global(P.gpu("U")), lay.to_global(U)
    assert np.isfinite(want).all()
    assert P.gm.counts()["nonfinite"] == 0
    assert np.isfinite(got).all() and (got[0] > 0).all() and (got[4] > 0).all()
    # both ends are at rest and uniform, so no mass leaves; 4096 additions of rounded terms
    assert abs(got[0].sum() / rho.sum() - 1) < 4096 * 2.0 ** -52
