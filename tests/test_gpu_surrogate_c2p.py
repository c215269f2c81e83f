"""The learned-guess closure that forms its table inputs from the conserved state and
writes the primitives in one kernel: blocks of unequal sizes with and without dual
energy, with the guesses of a network after one step of training (cells go to the queue and are
converted by the second kernel) and of a trained one (accepted cells), give the bits,
time steps and event counts of bisection."""
import numpy as np
import pytest

from paper_2609_37859_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_hydro import Pair, SCHEME_KEYS, tde, ctx, tables  # noqa: E402,F401


@pytest.mark.parametrize("train", [False, True])
@pytest.mark.parametrize("dual", [0, 1])
def test_fused_closure_equals_bisection(oracle, tde, ctx, tables, dual, train):
    net = tables[1]
    net.reset_weights_for_training()
    if train:
        net.train(seed=5, n_samples=1 << 18, epochs=6, batch=4096, lr=3e-3)
    else:
        net.train(seed=5, n_samples=1 << 12, epochs=1, batch=4096, lr=3e-3)
    rho0, v0 = 0.7382, 1.0948e8
    lay = wl.mixed_layout((16, 16, 8), 8, {(0, 0, 0), (1, 1, 0)},
                          ((-2.0, 2.0), (-2.0, 2.0), (-1.0, 1.0)), (0, 0, 0), 3)
    x, y, z = lay.cell_centres()
    r = np.sqrt(x ** 2 + y ** 2 + z ** 2)
    rho = 1e-6 + 1e-3 * np.exp(-((r - 1.0) / 0.3) ** 2)
    Pc = rho * rho0 * 1.380649e-16 * 1e4 / (0.6 * 1.6605e-24) / (rho0 * v0 * v0)
    W = wl.prim_state(lay, rho, -y * 0.3, x * 0.3, 0 * rho, Pc)
    scheme = dict(eos=1, recon=1, dual=dual, eta1=1e-3, eta2=1e-4, rho_floor=2e-6, p_floor=1e-13,
                  u_floor=1.5e-13, unit_rho=rho0, unit_e=v0 * v0)
    P = Pair(oracle, tde, ctx, lay, W, tables, **scheme)
    kw = {k: v for k, v in scheme.items() if k in SCHEME_KEYS}
    outs = {}
    for mode in ("INVERT_BISECT", "INVERT_SURROGATE"):
        P.gm.set_params(tde.make_params(eos_mode=getattr(tde, mode), **kw))
        P.gm.U.copy_(torch.from_numpy(P.U))
        P.gm.set_time(0.0)
        P.gm.counts(reset=True)
        dts = []
        for _ in range(2):
            dt = torch.zeros(1, dtype=torch.float64, device="cuda")
            P.gm.step(cfl=0.3, dt_out=dt)
            dts.append(float(dt))
        c = P.gm.counts()
        acc = c.pop("surrogate_accepted")
        outs[mode] = (P.gpu("U").copy(), dts, c, acc)
    b, s = outs["INVERT_BISECT"], outs["INVERT_SURROGATE"]
    assert np.array_equal(s[0], b[0]) and s[1] == b[1] and s[2] == b[2]
    # both routes are taken: accepted cells after training, queued ones without
    n = 4 * 16 * 16 * 8
    assert 0 < s[3] if train else s[3] < n
