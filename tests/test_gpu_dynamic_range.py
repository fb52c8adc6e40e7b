"""Column norms far outside the range whose squares are normal numbers, and non-finite values in every place
of a chunk: the right log|det M| and G, or the status, never a wrong number.

The oracle's pivoted QR scales its norms: on the shapes below its two orders of multiplication agree to 2e-15, and with
700-digit determinants where those were formed (4x4).  Tolerances are those of the parity tests.
"""
import numpy as np
import pytest

from tests.test_gpu_parity import G_ATOL, LD_RTOL, check_against_oracle, hq  # noqa: F401
from workloads import HolsteinParams, initial_fields, ordered_fields

pytestmark = pytest.mark.gpu

# (sides, beta, n_wrap, shift of one site's fields).  Long chains without a shift reach norms of 1e+-166 (beta = 90) and
# 1e+-277 (150); a raised site alone goes down to 1e-155 .. 1e-255, where squares are subnormal or zero, a lowered one
# up to 1e+146 .. 1e+239.  The sides cover panels of 32, 64, 128 and 256 rows.
RANGES = [(4, 4, 90.0, 10, 0.0), (4, 4, 150.0, 10, 0.0), (8, 8, 90.0, 10, 0.0), (10, 6, 95.0, 7, 0.0), (12, 12, 90.0, 10, 0.0),
          (4, 4, 16.0, 4, 15.6), (4, 4, 16.0, 4, 20.0), (4, 4, 16.0, 2, 25.0), (8, 8, 16.0, 4, 18.0), (10, 4, 16.0, 4, 16.7),
          (12, 8, 16.0, 4, 16.7), (4, 4, 16.0, 4, -15.6), (4, 4, 16.0, 4, -20.0), (4, 4, 16.0, 2, -25.0), (8, 8, 16.0, 4, -18.0)]


@pytest.mark.parametrize("nx,ny,beta,n_wrap,shift", RANGES)
def test_norms_beyond_the_range_of_their_squares(hq, nx, ny, beta, n_wrap, shift):  # noqa: F811
    import torch
    from oracle import dqmc
    p = HolsteinParams(nx=nx, ny=ny, beta=beta, n_wrap=n_wrap)
    X = ordered_fields(p, 1, 0.9)
    X[:, :, 5] += shift
    G_ref, ld_ref = dqmc.green_at(p, dqmc.kinetic_propagators(p)[0], X[0], 0)
    eng = hq.Engine(p, 1)
    eng.set_fields(X)
    _, ld = eng.log_weight()
    assert eng.observables()[0]["status"] == 0
    assert abs(ld[0] - ld_ref) <= LD_RTOL * abs(ld_ref)
    assert np.max(np.abs(eng.green(0) - G_ref)) < G_ATOL
    eng.close()
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    hq.logdet_noalloc(p, torch.from_numpy(X).cuda(), out)
    assert abs(out.item() - ld_ref) <= LD_RTOL * abs(ld_ref)


@pytest.mark.parametrize("local,method", [(True, 1), (False, 1), (False, 2)])
def test_sweeps_beyond_the_range_of_the_squares(hq, local, method):  # noqa: F811
    """Moves, two-sided G and block determinants where the chain's norms pass 1e+-166: the oracle's decisions."""
    p = HolsteinParams(nx=4, ny=4, beta=90.0, seed=21, block_method=method)
    check_against_oracle(hq, p, ordered_fields(p, 1, 0.9), 1, local=local, global_=not local)


def test_norms_beyond_64_bits_are_reported(hq):  # noqa: F811
    """Norms above 1e308 (beta = 180: 1e+-332) have no value in 64 bits."""
    p = HolsteinParams(nx=4, ny=4, beta=180.0)
    eng = hq.Engine(p, 1)
    eng.set_fields(ordered_fields(p, 1, 0.9))
    _, ld = eng.log_weight()
    assert not np.isfinite(ld[0]) and eng.observables()[0]["status"] == hq.HQ_ENAN
    eng.close()


@pytest.mark.parametrize("nx,ny", [(2, 2), (4, 4), (6, 4), (8, 8), (10, 10), (16, 16)])
def test_non_finite_values_in_every_place_of_a_chunk(hq, nx, ny):  # noqa: F811
    """The slice applied last in a chunk scales single rows, so that a value there reaches the factorisation in one row
    only; the one applied first is spread over every entry."""
    p = HolsteinParams(nx=nx, ny=ny, beta=0.8, n_wrap=4)
    X0 = initial_fields(p, 2)
    eng = hq.Engine(p, 2)
    eng.set_fields(X0)
    _, ld0 = eng.log_weight()
    eng.close()
    for slice_ in (0, 3, 4, 7):
        for site in (0, p.n_sites - 1):
            for value in (np.nan, -np.inf):  # exp(-dtau V) = NaN, inf
                X = X0.copy()
                X[1, slice_, site] = value
                eng = hq.Engine(p, 2)
                eng.set_fields(X)
                _, ld = eng.log_weight()
                where = (slice_, site, value)
                assert ld[0] == ld0[0] and not np.isfinite(ld[1]), where
                assert [o["status"] for o in eng.observables()] == [0, hq.HQ_ENAN], where
                assert np.isfinite(eng.green(0)).all() and not np.isfinite(eng.green(1)).all(), where
                eng.close()
