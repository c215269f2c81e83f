"""The edges of the EOS table in the fixed-point inversion: a density counts as on the table
up to half an FP64 ulp of log10 rho (of the axis's largest magnitude) beyond an edge, and as
clamped further out; and the lowest decade of the format."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

Q55 = np.longdouble(2.0) ** 55


def _eos(tde, lrho, le0=9.0):
    nr, nt = 4, 6
    le = le0 + np.add.outer(0.01 * np.arange(nr), 0.5 * np.arange(nt))
    return tde.EOS(tde.Context(0), nr, nt, lrho, (2.0, 4.0), le, 0.9 * le, 0.95 * le), le


@pytest.mark.parametrize("lrho", [(-14.0, 2.0), (-6.3, 1.7), (0.25, 0.75), (-0.9, 0.4), (3.0, 11.5), (-1.5, -0.1),
                                  (-30.1, 4.2), (-2.0, 2.0), (-7.9, -0.3), (1.1, 1.3), (-16.0, -3.7), (15.3, 33.3)])
def test_clamped_densities(lrho):
    from paper_2609_37859_gb300 import tde
    eos, _ = _eos(tde, lrho)
    # half an ulp of the larger edge's magnitude (at least 1), in log2 units of 2^-55
    m = max(1.0, abs(lrho[0]), abs(lrho[1]))
    tol = np.longdouble(np.spacing(m) / 2) * np.log2(np.longdouble(10)) * Q55
    near, far = [], []
    for edge, out in ((lrho[0], -1), (lrho[1], 1)):
        x = 10.0 ** edge
        lo = hi = x
        xs = [x]
        for _ in range(3 + int(40 * np.spacing(m) / np.spacing(1.0))):   # (an ulp of rho is 1 to 2 2^-53)
            lo, hi = np.nextafter(lo, 0.0), np.nextafter(hi, np.inf)
            xs += [lo, hi]
        for v in xs:
            d = out * (np.log10(np.longdouble(v)) - np.longdouble(edge)) * np.log2(np.longdouble(10)) * Q55
            # the logarithm and the edges are within two units each
            if d <= tol - 4:
                near.append(v)
            elif d >= tol + 4:
                far.append(v)
    assert near and far
    for rho, want in ((near, 0), (far, len(far))):
        r = torch.tensor(rho, dtype=torch.float64, device="cuda")
        c0 = eos.counts()["table_clamp"]
        eos.invert(r, torch.full_like(r, 1e10), P=torch.empty_like(r))
        assert eos.counts()["table_clamp"] - c0 == want


def test_lowest_decade_of_the_format(oracle):
    """Densities and energies between 10^-38 and 2^-126, which a table may still hold."""
    from paper_2609_37859_gb300 import tde
    lrho = (-37.99, -37.0)
    eos, le = _eos(tde, lrho, le0=-37.98)
    ot = oracle.EOSTable(le.shape[0], le.shape[1], lrho, (2.0, 4.0), le, 0.9 * le, 0.95 * le)
    rng = np.random.default_rng(3)
    rho = 10.0 ** rng.uniform(-37.98, -37.9, 400)
    e = 10.0 ** rng.uniform(-37.94, -37.0, 400)
    o = [torch.empty(400, dtype=torch.float64, device="cuda") for _ in range(3)]
    c = eos.invert(torch.from_numpy(rho).cuda(), torch.from_numpy(e).cuda(), T=o[0], P=o[1], cs2=o[2], counts=True)
    want = np.array([ot.invert(r, x) for r, x in zip(rho, e)])
    assert c.table_clamp == 0
    # FP64 logarithms of size 38 are off by at most 2^-48; 1e3 times that covers the slopes
    for k in range(3):
        assert np.abs(o[k].cpu().numpy() / want[:, k] - 1).max() < 4e-12
