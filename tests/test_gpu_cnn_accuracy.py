"""Error of F_cnn against 64 bits: rounding to nearest averages out over the points, a bias does not.

A sum of 432 products with FP32 roundings to nearest is off by about 2^-24 / sqrt(3) sqrt(432 / 2) = 5e-7 of its size
(standard deviation); F sums 16 channels of 40960 points, so the errors average to 6e-10 of the sum of the terms' sizes.  The
bound is three times that.
"""
import numpy as np
import pytest

from tests.test_gpu_parity import hq  # noqa: F401
from workloads import LARGEST, initial_fields

pytestmark = pytest.mark.gpu


def reference(p, theta, X):
    """(F, sum of the sizes of its terms) of every configuration from the FP32 inputs and bfloat16 weights, in 64 bits."""
    import torch
    from torch.nn.functional import conv3d, pad
    w1, b1, w2, b2, w3, b3 = torch.split(torch.from_numpy(theta.astype(np.float64)), [432, 16, 6912, 16, 432, 1])
    w1 = w1.reshape(3, 3, 3, 1, 16).permute(4, 3, 0, 1, 2)
    w2 = w2.reshape(3, 3, 3, 16, 16).permute(4, 3, 0, 1, 2)
    w3 = w3.reshape(27, 16).sum(0)
    z = (X + p.g / (p.mass * p.omega ** 2)).astype(np.float32).astype(np.float64)
    h = torch.from_numpy(z).reshape(-1, 1, p.n_slices, p.ny, p.nx)
    for w, b in ((w1, b1), (w2, b2)):
        h = torch.relu(conv3d(pad(h, (1, 1, 1, 1, 1, 1), mode="circular"), w, b))
    s = h.sum((2, 3, 4))
    return ((s * w3).sum(1) + p.n_slices * p.n_sites * b3).numpy(), (s * w3.abs()).sum(1).numpy()


def test_cnn_value_has_no_bias(hq):  # noqa: F811
    p = LARGEST
    errors = []
    for seed in range(6):
        X = initial_fields(p, 2, seed=seed)
        eng = hq.Engine(p, 2)
        eng.attach_network(1, 1)
        eng.set_params(hq.init_network(0))
        eng.cnn_set_params(hq.init_cnn(seed, out_scale=0.3))
        eng.set_fields(X)
        F = eng.cnn_eval()
        ref, size = reference(p, eng.cnn_get_params(bf16=True), X)
        errors.append((F - ref) / size)
        eng.close()
    assert np.sqrt(np.mean(np.square(errors))) < 2e-9
