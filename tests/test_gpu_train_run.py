"""Training runs by one cluster (batches up to 12,288) and by the per-step
kernels (larger ones) against the FP64 replica: batches that leave half-warps
idle, fill them unevenly, need a second fetch of samples, and lie on both
sides of the line."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


# FP32 rounding of the gradients moves a weight by a few 1e-6 a step of Adam
# (each at most the learning rate, 3e-3): 5e-4 over six steps, as the
# twelve-step test allows 2e-4 at a batch of 512
@pytest.mark.parametrize("batch", [1, 37, 511, 513, 1025, 8193, 12288, 12289])
def test_six_steps_match_the_replica(gpu_lib, batch):
    B = gpu_lib
    tp = B.make_train_params(n_samples=20_011, batch=batch, steps=6, lr0=3e-3, lr_min=1e-4, tol=1e30, seed=91)
    h = B.ph_mlp_train(tp, 1.0, 4.5)
    w, _, loss = B.ph_mlp_get(h)
    ref, losses = M.train(4.5, 20_011, batch, 6, 3e-3, 1e-4, seed=91)
    np.testing.assert_allclose(w, ref, atol=5e-4)
    assert abs(loss - losses[-1]) <= 1e-3 * abs(losses[-1]) + 1e-9
    B.ph_free(h)
