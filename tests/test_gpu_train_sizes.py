"""Training with fewer samples than a batch: no step is taken, the weights stay, and the
report says so."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_fewer_samples_than_a_batch():
    from paper_2609_37859_gb300 import tde
    eos = tde.EOS.from_file(tde.Context(0), os.path.join(os.path.dirname(tde.__file__), "data", "eos_saha_hhe_256.npz"))
    eos.train(seed=3, n_samples=4096, epochs=1, batch=1024)
    w = eos.get_weights()
    r = eos.train(seed=3, n_samples=512, epochs=2, batch=1024)
    assert r["batches"] == 0 and r["loss_first"] == 0.0 and r["loss_last"] == 0.0
    assert np.array_equal(eos.get_weights(), w)
