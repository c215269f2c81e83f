"""The column form of the remap at the edges of its range: width ratios up to just
below two and just above, offsets that put samples on source centres, targets
reaching past an outflow source, periodic wraps, odd and one-cell blocks; and no
neighbour's NaN in a cell that does not sample it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from parity import assert_parity  # noqa: E402
from paper_2609_37859_gb300 import workloads as wl  # noqa: E402
from test_gpu_hydro import tde, ctx  # noqa: E402,F401
from test_gpu_remap import Side, TOL, remap_both  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("N,half", [((17, 9, 33), 0.5), ((40, 24, 20), 1.0), ((21, 21, 21), 1.3),
                                    ((16, 16, 16), 0.999), ((16, 16, 16), 1.001), ((48, 5, 1), 0.7),
                                    ((30, 31, 29), 0.03)])
def test_matches_oracle(oracle, tde, ctx, N, half, bc):
    src = wl.uniform_layout((16, 16, 16), (8, 8, 8), ((-0.5, 0.5),) * 3, bc=(bc,) * 3, ng=2)
    dom = tuple((-half + 0.01 * a, half + 0.01 * a) for a in range(3))
    dst = wl.uniform_layout(N, (7, 8, 9), dom, bc=(0, 0, 0), ng=2)
    S, D = Side(oracle, tde, ctx, src, 1), Side(oracle, tde, ctx, dst, 1)
    U = S.om.prim_to_cons(wl.random_smooth(src, seed=9, drho=0.4))
    got, want = remap_both(oracle, tde, S, D, U, tde.REMAP_THERMAL)
    assert_parity(got, want, TOL)   # the remap tests' bound


def test_a_bad_source_cell_stays_local(oracle, tde, ctx):
    src = wl.uniform_layout((16, 16, 16), (8, 8, 8), ((-0.5, 0.5),) * 3, bc=(0, 0, 0), ng=2)
    dst = wl.uniform_layout((32, 32, 32), (16, 16, 16), ((-0.75, 0.75),) * 3, bc=(0, 0, 0), ng=2)
    S, D = Side(oracle, tde, ctx, src, 1), Side(oracle, tde, ctx, dst, 1)
    G = src.to_global(S.om.prim_to_cons(wl.random_smooth(src, seed=9)))
    G[:, 0, 0, 0] = np.nan
    S.gm.U.copy_(torch.from_numpy(src.from_global(G)))
    D.gm.U.zero_()
    D.gm.remap_from(S.gm, S.gm.U, tde.REMAP_THERMAL)
    got = dst.to_global(D.gm.U.cpu().numpy())
    bad = np.argwhere(~np.isfinite(got[0]))
    # a sample reaches two source cells along a direction, a target cell spans 3/4 of one
    x = -0.75 + (bad + 0.5) * 1.5 / 32
    assert bad.size and np.abs(x + 0.5 - 0.5 / 16).max() <= 1.5 / 16
    assert np.isfinite(got[0][:3]).all() and np.isfinite(got[0][:, :3]).all() and np.isfinite(got[0][:, :, :3]).all()
