"""Edges of the tensor-core products, panels and correction vectors, through the engine against the oracle.

The shapes cross the sizes at which the kernels change form: panels of 4 to 16 columns and 32, 64, 128,
256 rows, matrices of 16 (FP64 products), 64 (one accumulator) and more rows, one, two or four matrix
columns per kinetic tile, correction vectors with an odd number of slices, chunks longer than one
16-term step and shorter last chunks.  Tolerances are those of the parity tests: FP64 results to 1e-10,
decisions (fields) bit for bit under the shared Philox stream.
"""
import numpy as np
import pytest

from tests.test_gpu_parity import check_against_oracle, hq  # noqa: F401
from workloads import HolsteinParams, initial_fields, random_fields

pytestmark = pytest.mark.gpu


# (sides, beta, n_wrap): N = 4 .. 256 over every panel height and tile form
SHAPES = [(2, 2, 0.9, 4), (4, 2, 1.1, 3), (4, 4, 1.3, 5), (6, 2, 0.7, 3), (4, 6, 1.0, 10), (8, 4, 0.9, 4), (2, 16, 0.8, 4),
          (6, 8, 0.6, 5), (10, 4, 0.7, 3), (8, 8, 0.5, 5), (12, 6, 0.5, 2), (10, 10, 0.4, 3), (16, 8, 0.4, 4),
          (12, 12, 0.4, 4), (16, 12, 0.3, 3), (14, 16, 0.3, 2), (16, 16, 0.3, 2)]


@pytest.mark.parametrize("nx,ny,beta,n_wrap", SHAPES)
def test_weight_and_green_over_all_forms(hq, nx, ny, beta, n_wrap):  # noqa: F811
    from oracle import dqmc
    p = HolsteinParams(nx=nx, ny=ny, beta=beta, n_wrap=n_wrap)
    X = random_fields(p, 2, seed=nx + 31 * ny, scale=1.0, offset=-1.2)
    eng = hq.Engine(p, 2)
    eng.set_fields(X)
    _, ld = eng.log_weight()
    expK, _ = dqmc.kinetic_propagators(p)
    for c in range(2):
        G_ref, ld_ref = dqmc.green_at(p, expK, X[c], 0)
        assert abs(ld[c] - ld_ref) <= 1e-10 * abs(ld_ref)
        assert np.max(np.abs(eng.green(c) - G_ref)) < 1e-10
    eng.close()


# odd L with several chains (every chain's vectors stay aligned), n_wrap above 16, a last chunk of one slice
@pytest.mark.parametrize("nx,ny,beta,n_wrap,method", [(4, 4, 0.7, 3, 2), (6, 4, 1.9, 18, 2), (8, 6, 1.1, 5, 2), (10, 2, 0.9, 4, 2),
                                                      (8, 8, 0.7, 6, 2), (4, 6, 1.9, 18, 1), (2, 2, 0.5, 2, 2)])
def test_block_moves_over_all_forms(hq, nx, ny, beta, n_wrap, method):  # noqa: F811
    p = HolsteinParams(nx=nx, ny=ny, beta=beta, n_wrap=n_wrap, delay_k=16, seed=900 + nx * ny, block_method=method)
    check_against_oracle(hq, p, initial_fields(p, 3, seed=8), 2)


# delayed-update ranks around the 16-term step, with the vectors in shared and (k = 32, N = 256) global memory
@pytest.mark.parametrize("nx,ny,k", [(16, 16, 32), (12, 10, 17), (6, 6, 15), (2, 4, 32)])
def test_local_moves_over_delay_ranks(hq, nx, ny, k):  # noqa: F811
    p = HolsteinParams(nx=nx, ny=ny, beta=0.3, n_wrap=2, delay_k=k, seed=500 + k)
    check_against_oracle(hq, p, initial_fields(p, 2, seed=4), 1, global_=False)


def test_non_finite_fields_are_reported(hq):  # noqa: F811
    """A NaN field reaches log|det M| and the status through the fixed-point splits; other chains are untouched."""
    for side in (4, 8, 10):
        p = HolsteinParams(nx=side, ny=side, beta=0.8, n_wrap=4)
        X = initial_fields(p, 2)
        eng = hq.Engine(p, 2)
        eng.set_fields(X)
        _, ld0 = eng.log_weight()
        X[1, 3, 1] = np.nan
        eng.set_fields(X)
        _, ld = eng.log_weight()
        assert ld[0] == ld0[0] and not np.isfinite(ld[1])
        obs = eng.observables()
        assert obs[0]["status"] == 0 and obs[1]["status"] == hq.HQ_ENAN
        eng.close()


# (sides, beta, batch): tiles of 16 points with a remainder, one and several CTAs per sample, more samples
# than are trained at a time (two rounds), blocks of 128 points with a remainder.  The convolutional gradient
# is FP32 (sums of up to 432 products: 432 * 2^-24 = 3e-5); the patch gradient keeps 16 bits of an activation
# and has the parity tests' tolerance.
@pytest.mark.parametrize("nx,ny,beta,batch", [(4, 4, 0.5, 1), (6, 4, 0.7, 3), (4, 4, 0.5, 155), (10, 4, 0.6, 9), (6, 6, 1.1, 40)])
def test_gradients_over_all_splits(hq, nx, ny, beta, batch):  # noqa: F811
    import torch
    from oracle import cnn, nn
    p = HolsteinParams(nx=nx, ny=ny, beta=beta)
    X = random_fields(p, batch, seed=5 * nx + ny, offset=-1.4)
    y = np.linspace(-3.0, 2.0, batch)
    eng = hq.Engine(p, 1)
    eng.attach_network(batch, batch)
    tp, tc = nn.init_params(2).astype(np.float32) * np.float32(3.0), cnn.init_params(3, out_scale=30.0)
    eng.set_params(tp)
    eng.cnn_set_params(tc)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    g, loss = eng.cnn_gradient(Xd, yd)
    lref, gref = cnn.loss_and_grad(p, nn.to_bfloat16(tc.astype(np.float32)), X, y)
    assert abs(loss - lref) <= 1e-4 * lref
    assert np.max(np.abs(g - gref)) <= 1e-4 * np.max(np.abs(gref))
    g, loss = eng.nn_gradient(Xd, yd)
    lref, gref = nn.loss_and_grad(p, nn.to_bfloat16(tp), X, y)
    assert abs(loss - lref) <= 2e-3 * lref
    assert np.max(np.abs(g - gref)) <= 2e-3 * np.max(np.abs(gref))
    eng.close()
