"""Training where the cooperative launch is refused, as where a process is not
given every SM: the call goes on with three launches per mini-batch and gives
the same training.  Two trainings that each follow FP64 Adam to 1e-3 k lr after k
steps (the bound of the training tests) differ by at most twice that, their
losses by twice 1e-4.  FLBM_INJECT_REFUSE=1 refuses the launch on the host."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# one batch, whole and ragged epochs, more batches than one launch takes, a
# batch of several tiles per CTA
@pytest.mark.parametrize("n,batch,epochs", [(5, 8, 3), (1000, 96, 2), (5000, 1300, 2), (1100, 1, 1), (40000, 19456, 2)])
def test_training_goes_on_without_a_cooperative_launch(monkeypatch, n, batch, epochs):
    import torch

    from oracle import mlp as M
    from paper_2601_03806_gb300 import flbm
    rng = np.random.default_rng(n)
    theta0 = (M.init_params(3) + 0.05 * rng.normal(size=M.NPARAM)).astype(np.float32)
    x, t = (torch.from_numpy(rng.normal(size=(n, k)).astype(np.float32)).cuda() for k in (28, 27))
    lr = 1e-3
    a, la = flbm.mlp_train(theta0, x, t, epochs=epochs, batch=batch, lr=lr, seed=5)
    monkeypatch.setenv("FLBM_INJECT_REFUSE", "1")
    b, lb = flbm.mlp_train(theta0, x, t, epochs=epochs, batch=batch, lr=lr, seed=5)
    again, _ = flbm.mlp_train(theta0, x, t, epochs=epochs, batch=batch, lr=lr, seed=5)
    steps = epochs * -(-n // min(batch, n))
    assert np.sqrt(np.mean((a - b).astype(float) ** 2)) <= 2e-3 * steps * lr
    assert np.abs(la - lb).max() <= 2e-4 * la.max()
    assert np.array_equal(b, again)
    assert not np.array_equal(a, theta0)
