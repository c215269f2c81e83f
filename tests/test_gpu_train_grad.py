"""The training gradient at partial CTAs (counts around multiples of 32 samples) and
into a gradient buffer that starts on any float."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_surrogate import NP, bf16_round, dev, env, random_weights, tde  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(1, 0), (31, 1), (32, 2), (33, 3), (4096, 0), (4129, 1)])
def test_gradient_matches_oracle(tde, oracle, env, n, shift):
    _, eos, _ = env
    w = random_weights(4)
    eos.set_weights(w)
    rng = np.random.default_rng(n)
    x = rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    t = rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    g = torch.zeros(NP + shift, dtype=torch.float32, device="cuda")[shift:]
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    eos.grad(dev(x), dev(t), g, loss)
    torch.cuda.synchronize()
    lo, go = oracle.mlp_loss_grad(bf16_round(w), x.astype(np.float64), t.astype(np.float64))
    # FP32 sums of at most 64 + n terms with __expf's few ulps: below 1e-4 relative
    # in norm (the bound of the training test is ten times this)
    assert float(loss) == pytest.approx(lo, rel=1e-4)
    assert np.linalg.norm(g.cpu().numpy() - go) <= 1e-4 * np.linalg.norm(go)
