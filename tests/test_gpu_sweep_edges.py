"""The sweep kernel at the edges of its chunks (8 FP64, 16 FP32 steps) and
bands (32 rows): widths below, at and above one and two chunks and the 31
steps of the lanes' skew, heights around whole bands, more units than warps.

Tolerance: each cell's value rounds a few times per step of a chain of at
most nx + ny cells, sums of K <= 84 terms: below (nx + ny + K) 2^-53 < 1e-13 of
the largest value in FP64; 2^-24 in place of 2^-53 gives 4e-5 in FP32.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,order", [(1, 33, 4), (7, 64, 4), (8, 32, 6), (9, 31, 4), (16, 65, 4), (17, 1, 4),
                                         (30, 96, 4), (31, 32, 4), (32, 34, 6), (33, 63, 4), (47, 40, 4),
                                         (64, 33, 4), (39, 161, 4), (40, 700, 12)])
@pytest.mark.parametrize("fp32", [False, True])
def test_transport_sweep(nx, ny, order, fp32):
    import torch
    from paper_2507_03975_gb300 import gsis
    p = W.random_problem(nx, ny, order=order, seed=3 * nx + ny)
    rho = np.random.default_rng(nx).uniform(0.0, 2.0, p.N)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    opt = gsis.default_options(precision=gsis.FP32_SWEEP if fp32 else gsis.FP64)
    r = gsis.transport_sweep(p.dx, p.dy, p.mu, p.eta, p.w, t(p.sigma_a), t(p.sigma_s), t(p.q), t(rho),
                             t(p.inflow.reshape(-1)), opt)
    o = oracle.transport_sweep(p, rho)
    tol = (4e-5 if fp32 else 1e-13) * np.abs(o["rho"]).max()
    for k, v in (("rho", o["rho"]), ("F", np.concatenate([o["Fx"], o["Fy"]])), ("bflux", o["fb"])):
        assert np.abs(r[k].cpu().numpy() - v).max() <= tol, k


@pytest.mark.parametrize("nx,ny,order", [(1, 1, 4), (2, 33, 4), (3, 31, 4), (17, 32, 6), (18, 40, 4), (19, 64, 4),
                                         (194, 133, 16), (195, 150, 16)])
def test_reciprocal_tiles(nx, ny, order):
    """Widths at which nx + 62 columns fill, just miss or just exceed the
    reciprocal table's tiles of 16 and (the last two) 64 columns."""
    test_transport_sweep(nx, ny, order, False)
