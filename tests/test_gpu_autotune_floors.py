"""The sweep autotuner on a state whose update reaches the floors and holds a bad cell: its
sweeps count such events as any sweep does, and the counters and the state are as before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_37859_gb300 import workloads as wl  # noqa: E402
from test_gpu_hydro import Pair, tde, ctx, tables  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eos", [0, 1])
def test_counters_are_put_back(oracle, tde, ctx, tables, eos):
    lay = wl.uniform_layout((16, 16, 16), (8, 8, 8), bc=(1, 1, 1), ng=3)
    one = np.ones((16, 16, 16))
    W = wl.prim_state(lay, 1e-8 * one, 0 * one, 0 * one, 0 * one, one)
    floors = dict(rho_floor=1e-10, p_floor=1e-12, u_floor=1e-12)
    P = Pair(oracle, tde, ctx, lay, W, tables if eos else None, eos=eos, recon=1, dual=1, eta1=1e-3, eta2=1e-4, **floors)
    G = lay.to_global(P.U)
    G[0, 3, 4, 5] = 1e-12          # below the density floor
    G[5, 8, :, :] = 1e-14          # auxiliary energies below theirs
    G[1, 12, 12, 12] = np.nan
    U = lay.from_global(G)
    P.gm.U.copy_(torch.from_numpy(U))
    P.gm.compute_dt(0.3, torch.zeros(lay.nb, dtype=torch.float64, device="cuda"))   # (counts on its own)
    before = P.gm.counts()
    P.gm.autotune(reps=2)
    torch.cuda.synchronize()
    assert P.gm.counts() == before
    assert np.array_equal(P.gpu("U"), U, equal_nan=True)
