"""Neighbouring cells whose differences lie at the bottom of the FP64 range (a blast
wave's precursor in gas at rest): their products underflow and the sum of two has no
finite reciprocal.  The reconstruction stays finite there and agrees with the oracle.
Unit density and pressure, so a stage's tolerance of 1e-12 per cell holds absolutely."""
import numpy as np
import pytest

from paper_2609_37859_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_hydro import Pair, STAGE_TOL, tde, ctx  # noqa: E402,F401


@pytest.mark.parametrize("amp", [1e-323, 1e-310, 2e-309, 1e-308, 1e-200, 1e-160])
@pytest.mark.parametrize("recon,riemann,block", [(0, 0, 16), (0, 1, 16), (1, 1, 16), (0, 1, 32), (0, 0, 5)])
def test_step_with_tiny_velocity_differences(oracle, tde, ctx, amp, recon, riemann, block):
    n = 2 * block
    lay = wl.uniform_layout((n, block, block), (block,) * 3, bc=(0, 0, 0), ng=3 if recon else 2)
    x, y, z = lay.cell_centres()
    v = amp * np.round(n * (x + 2 * y + 3 * z))   # a ramp along each direction
    one = np.ones_like(v)
    P = Pair(oracle, tde, ctx, lay, wl.prim_state(lay, one, v, -v, 2 * v, one), recon=recon, riemann=riemann, dual=1,
             eta1=1e-3, eta2=1e-4)
    U = P.U.copy()
    d = P.om.cfl_dt(U, 0.3).min()
    P.om.step(U, d, 0.0)
    P.gm.step(cfl=0.3)
    G, O = lay.to_global(P.gpu("U")), lay.to_global(U)
    assert np.isfinite(O).all() and np.isfinite(G).all()
    assert np.abs(G - O).max() <= STAGE_TOL
