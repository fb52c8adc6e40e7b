"""G where the rows of the stabilised product's triangular factor differ in size by orders of magnitude.

A lowered site makes its row of every slice product large; the triangular factors' rows and columns spread with it,
and G depends on their small entries.  The oracle factors every second product (error 6e-15 here against a
420-digit inverse); FP64 products in the engine's order of operations reach 1e-12 to 2e-11, so the parity tests' 1e-10 holds
for any product that keeps the small entries.
"""
import numpy as np
import pytest

from tests.test_gpu_parity import G_ATOL, LD_RTOL, hq  # noqa: F401
from workloads import HolsteinParams, ordered_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,beta,n_wrap,shift", [(8, 8, 16.0, 10, -6.0), (8, 8, 16.0, 10, -10.0), (8, 8, 16.0, 4, -14.0),
                                                     (10, 6, 8.0, 10, -6.0), (12, 12, 4.0, 10, -6.0), (6, 4, 16.0, 10, -6.0)])
def test_green_of_a_lowered_site(hq, nx, ny, beta, n_wrap, shift):  # noqa: F811
    from oracle import dqmc
    p = HolsteinParams(nx=nx, ny=ny, beta=beta, n_wrap=n_wrap)
    X = ordered_fields(p, 1, 0.9)
    X[:, :, 5] += shift
    G_ref, ld_ref = dqmc.green_at(p, dqmc.kinetic_propagators(p)[0], X[0], 0, n_wrap=2)
    eng = hq.Engine(p, 1)
    eng.set_fields(X)
    _, ld = eng.log_weight()
    assert abs(ld[0] - ld_ref) <= LD_RTOL * abs(ld_ref)
    assert np.max(np.abs(eng.green(0) - G_ref)) < G_ATOL
    eng.close()
