"""The column form of the remap with each run length along z that a target's size leads to
(1 to 32 cells a thread), also where a run ends inside a block; small blocks, whose runs are
shortened; and a target of one plane (a thread per cell)."""
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


@pytest.mark.parametrize("N,block", [((17, 9, 33), 17), ((49, 50, 51), 25), ((64, 64, 70), 32), ((100, 100, 100), 20),
                                     ((128, 128, 129), 32), ((160, 161, 160), 32), ((64, 64, 264), 8),
                                     ((300, 200, 1), 32), ((200, 1, 200), 32)])
def test_matches_oracle(oracle, tde, ctx, N, block):
    src = wl.uniform_layout((32, 32, 32), (16, 16, 16), ((-0.5, 0.5),) * 3, bc=(1, 1, 1), ng=2)
    dst = wl.uniform_layout(N, tuple(min(block, n) for n in N), ((-0.5, 0.5), (-0.45, 0.55), (-0.5, 0.43)), bc=(0, 0, 0), ng=2)
    if 1 in N:   # (a flat target of its own width samples a flat source)
        flat = tuple(32 if n > 1 else 1 for n in N)
        src = wl.uniform_layout(flat, tuple(min(16, n) for n in flat), ((-0.5, 0.5),) * 3, bc=(1, 1, 1), ng=2)
    S, D = Side(oracle, tde, ctx, src, 1), Side(oracle, tde, ctx, dst, 1)
    U = S.om.prim_to_cons(wl.random_smooth(src, seed=9, drho=0.4))
    got, want = remap_both(oracle, tde, S, D, U, tde.REMAP_THERMAL)
    assert_parity(got, want, TOL)   # the remap tests' bound


@pytest.mark.parametrize("N,half", [((40, 40, 40), 0.5), ((21, 21, 21), 0.5), ((16, 16, 16), 0.46875), ((64, 20, 20), 0.5)])
def test_an_infinite_source_cell(oracle, tde, ctx, N, half):
    """Target cells that sample an infinite density have an infinite density, as the sum of
    the used entries gives it; the others are untouched."""
    src = wl.uniform_layout((16, 16, 16), (8, 8, 8), ((-0.5, 0.5),) * 3, bc=(0, 0, 0), ng=2)
    dst = wl.uniform_layout(N, (8, 8, 8), ((-half, half),) * 3, bc=(0, 0, 0), ng=2)
    S, D = Side(oracle, tde, ctx, src, 1), Side(oracle, tde, ctx, dst, 1)
    G = src.to_global(S.om.prim_to_cons(wl.random_smooth(src, seed=9)))
    G[0, 5, 7, 9] = np.inf
    with np.errstate(invalid="ignore"):
        got, want = remap_both(oracle, tde, S, D, src.from_global(G), tde.REMAP_THERMAL)
    assert np.isinf(got[0]).any() and np.array_equal(np.isposinf(got[0]), np.isposinf(want[0]))
    assert not np.isnan(got[0]).any() and not np.isnan(want[0]).any()
