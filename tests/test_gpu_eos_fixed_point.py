"""The fixed-point EOS inversion against the oracle on tables of odd shapes, at the
edges of its cells and of the table, and where a table leaves the fixed-point
format (FP64 route)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _table(rng, nr, nt, shift):
    """Columns increasing in T with uneven cells (0.02 to 0.3 dex), rows that differ."""
    le = np.cumsum(rng.uniform(0.02, 0.3, (nr, nt)), axis=1) + rng.uniform(-0.5, 0.5, (nr, 1)) + shift
    lp = 0.9 * le + rng.uniform(-0.01, 0.01, (nr, nt))
    lc = 1.1 * le + rng.uniform(-0.01, 0.01, (nr, nt))
    return le, lp, lc


# (2, 2): one cell; (3, 90), (65, 2), (40, 33): odd shapes; a shift of +37 puts
# entries beyond the format (|log10| >= 38), one of -12 makes them negative; the
# fixed-point path and the bucket search are taken by the others
@pytest.mark.parametrize("nr,nt,shift", [(2, 2, 3.0), (3, 90, -12.0), (65, 2, 0.0), (40, 33, 9.0), (5, 8, 37.0)])
def test_inversion_matches_the_oracle(oracle, nr, nt, shift):
    from paper_2609_37859_gb300 import tde
    rng = np.random.default_rng(nr * 1000 + nt)
    le, lp, lc = _table(rng, nr, nt, shift)
    lrho, lT = (-6.3, 1.7), (1.0, 6.0)
    ot = oracle.EOSTable(nr, nt, lrho, lT, le, lp, lc)
    gt = tde.EOS(tde.Context(0), nr, nt, lrho, lT, le, lp, lc)
    n = 6000
    lr = rng.uniform(lrho[0] - 0.3, lrho[1] + 0.3, n)
    ly = rng.uniform(le.min() - 0.3, le.max() + 0.3, n)
    # on nodes and density grid lines, and a rounding away from them
    k = n // 3
    i, j = rng.integers(0, nr, k), rng.integers(0, nt, k)
    lr[:k] = lrho[0] + i * (lrho[1] - lrho[0]) / (nr - 1)
    ly[:k] = le[i, j]
    rho, e = 10.0 ** lr, 10.0 ** ly
    step = rng.integers(-2, 3, k)
    e[:k] = np.where(step > 0, np.nextafter(e[:k], np.inf), np.where(step < 0, np.nextafter(e[:k], 0), e[:k]))
    e[-6:] = [0.0, -1.0, 1e-310, 1e300, np.inf, 1e-300]
    rho[-12:-6] = [0.0, -1.0, 1e-310, 1e300, np.inf, 1e-300]
    want = np.array([ot.invert(r, x) for r, x in zip(rho, e)])
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    outs = []
    for mode in (tde.INVERT_BISECT, tde.INVERT_BISECT_PLAIN):
        o = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3)]
        gt.invert(d(rho), d(e), T=o[0], P=o[1], cs2=o[2], mode=mode)
        outs.append([x.cpu().numpy() for x in o])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)   # the cell is unique, so the search does not matter
    # The oracle's FP64 logarithms (size below 64) are off by at most 2^-48, the
    # position in a cell of at least 0.02 dex by 100 times that, times a cell's
    # 0.4 dex in the results and ln 10: 3.3e-13; T's cell of up to 5 dex: 4.1e-12.
    cell_T = (lT[1] - lT[0]) / (nt - 1)
    for got, col, tol in ((outs[0][0], 0, 1e-13 + 8.2e-13 * cell_T), (outs[0][1], 1, 5e-13), (outs[0][2], 2, 5e-13)):
        assert np.max(np.abs(got / want[:, col] - 1)) < tol
