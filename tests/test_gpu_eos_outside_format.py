"""Tables with an entry outside the fixed-point format (|log10| of 38 or more): every search
form gives the same bits, on and beside the nodes too, the learned form settles cells by its
Newton step as on other tables, and the time step without allocations equals the mesh's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_37859_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu

NR, NT, LRHO, LT = 40, 60, (-6.0, 2.0), (1.0, 6.0)


def _arrays(which):
    x, y = np.meshgrid(np.linspace(0, 1, NR), np.linspace(0, 1, NT), indexing="ij")
    le = 8.0 + 6.0 * y + 0.3 * np.sin(5 * x) + 0.2 * np.sin(9 * y)
    lp = 0.9 * le - 1.0 + x
    lc = 0.95 * le
    if which == "one":        # a single entry, in a corner no input comes near
        lc[NR - 1, NT - 1] = 38.5
    elif which == "inner":    # away from the corners
        lc[20, 30] = 38.5
        lp[5:9, 40:50] += 40.0
        le[30, 50:] += 30.0
    elif which == "P":
        lp = lp + 40.0
    elif which == "half":     # the hot half of the columns
        le = 3.2 * le
    return le, lp, lc


@pytest.mark.parametrize("which", ["one", "inner", "P", "half"])
def test_all_forms_agree(which):
    from paper_2609_37859_gb300 import tde
    le, lp, lc = _arrays(which)
    eos = tde.EOS(tde.Context(0), NR, NT, LRHO, LT, le, lp, lc)
    eos.train(seed=4, n_samples=1 << 16, epochs=10, batch=2048)
    rng = np.random.default_rng(8)
    n = 40000
    lr, ly = rng.uniform(LRHO[0] - 0.2, LRHO[1] + 0.2, n), rng.uniform(le.min() - 0.2, le.max() + 0.2, n)
    i, j = rng.integers(0, NR, n // 2), rng.integers(0, NT, n // 2)
    lr[: n // 2] = LRHO[0] + i * (LRHO[1] - LRHO[0]) / (NR - 1)   # nodes, and up to three roundings beside them
    ly[: n // 2] = le[i, j]
    e = 10.0 ** ly
    e[: n // 2] += rng.integers(-3, 4, n // 2) * np.spacing(e[: n // 2])
    rho, e = torch.from_numpy(10.0 ** lr).cuda(), torch.from_numpy(e).cuda()
    outs = []
    for mode in (tde.INVERT_BISECT, tde.INVERT_BISECT_PLAIN, tde.INVERT_SURROGATE):
        c0 = eos.counts()
        o = [torch.full((n,), -1.0, dtype=torch.float64, device="cuda") for _ in range(3)]
        eos.invert(rho, e, T=o[0], P=o[1], cs2=o[2], mode=mode)
        c1 = eos.counts()
        outs.append((o, c1["table_clamp"] - c0["table_clamp"], c1["surrogate_accepted"] - c0["surrogate_accepted"]))
    for o, clamp, _ in outs[1:]:
        assert clamp == outs[0][1]
        for a, b in zip(o, outs[0][0]):
            assert torch.equal(a, b)
    assert [x[2] for x in outs[:2]] == [0, 0] and outs[2][2] > 0


@pytest.mark.parametrize("which", ["in", "one", "inner", "P", "half"])
def test_noalloc_dt_has_the_same_bits(which):
    from paper_2609_37859_gb300 import tde
    ctx = tde.Context(0)
    arrs = _arrays(which)
    eos = tde.EOS(ctx, NR, NT, LRHO, LT, *arrs)
    table = (NR, NT, LRHO, LT) + tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrs)
    lay = wl.uniform_layout((32, 24, 16), (8, 8, 8), bc=(1, 0, 1), ng=2)
    p = tde.make_params(eos=1, dual=1, rho_floor=1e-30, p_floor=1e-30, u_floor=1e-30)
    m = tde.Mesh(ctx, lay, p, eos)
    rng = np.random.default_rng(2)
    U = np.zeros((6, lay.ntot))
    U[0] = 10 ** rng.uniform(LRHO[0], LRHO[1], lay.ntot)
    U[4] = U[0] * 10 ** rng.uniform(arrs[0].min(), arrs[0].max(), lay.ntot)
    U[1] = 0.1 * np.sqrt(U[0] * U[4])
    U[5] = U[4]
    m.U.copy_(torch.from_numpy(U))
    got, want = (torch.zeros(lay.nb, dtype=torch.float64, device="cuda") for _ in range(2))
    for _ in range(2):
        m.compute_dt(0.3, want)
        tde.compute_dt_noalloc(ctx, lay, p, m.U, 0.3, dt_block=got, table=table)
        assert torch.isfinite(want).all() and torch.equal(got, want)
