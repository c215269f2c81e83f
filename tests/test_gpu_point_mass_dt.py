"""The point mass's time-step limit in cold gas, where it sets every block's step:
positions inside a block, beside it, on cell centres, faces and midpoints, with and
without excision and softening, in blocks down to one cell wide.  The CFL pass takes a
far block's limit from the cells nearest to the point mass; the allocation-free entry
point evaluates every cell.  Both give the same bits, the oracle's values to 1e-14."""
import numpy as np
import pytest

from paper_2609_37859_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_hydro import Pair, SCHEME_KEYS, tde, ctx  # noqa: E402,F401

POS = [(0.5, 0.5, 0.5), (0.53125, 0.46875, 0.28125), (0.51, 0.77, 0.13), (-0.2, 0.5, 1.3), (0.25, 0.53125, 3.0),
       (1e3, -1e3, 2e3)]


@pytest.mark.parametrize("pos", POS)
@pytest.mark.parametrize("N,block", [((16, 16, 16), (8, 8, 8)), ((17, 9, 5), (4, 8, 4)), ((32, 32, 32), (32, 32, 32))])
@pytest.mark.parametrize("r_soft,r_exc", [(0.05, 0.0), (0.0, 0.12), (0.4, 0.3)])
def test_dt_of_cold_gas_is_the_point_mass_limit(oracle, tde, ctx, pos, N, block, r_soft, r_exc):
    lay = wl.uniform_layout(N, block, bc=(1, 0, 1), ng=2)
    bh = dict(on=1, excise=int(r_exc > 0), GM=0.3, r_soft=r_soft, r_exc=r_exc, x0=pos)
    one = np.ones((N[2], N[1], N[0]))
    scheme = dict(p_floor=1e-30)
    P = Pair(oracle, tde, ctx, lay, wl.prim_state(lay, one, 0 * one, 0 * one, 0 * one, 1e-20 * one), bh=bh, **scheme)
    want = P.om.cfl_dt(P.U, 0.35)
    dtb = torch.zeros(P.nb, dtype=torch.float64, device=P.dev)
    dmin = torch.zeros(1, dtype=torch.float64, device=P.dev)
    P.gm.compute_dt(0.35, dtb, dmin, t_block=P.dvec(0.0), bh=P.bh)
    got = dtb.cpu().numpy()
    assert np.isfinite(got).all() and (got < 1e8).all()   # not the hydro limit's 1e9
    assert np.allclose(got, want, rtol=1e-14, atol=0)
    full = torch.zeros_like(dtb)
    tde.compute_dt_noalloc(ctx, lay, tde.make_params(**scheme), P.gm.U, 0.35, full, torch.zeros_like(dmin), bh=P.bh)
    assert np.array_equal(got, full.cpu().numpy())
