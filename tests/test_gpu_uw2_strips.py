"""The second-order residual kernel at the edges of its strips' width (29
columns) and over several strips of 16 rows, with and without the limiter, on
a non-uniform mesh with inflow.

Tolerance: the kernel's operations are the oracle's up to the order of a few
roundings; two iterations of the scheme amplify 1e-16 by less than 1e4 on
these meshes: 1e-11 of the largest value is asked (FP32: 1e-5).
"""
import numpy as np
import pytest

import workloads as W
from oracle import uw2 as oracle_uw2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,order", [(1, 1, 4), (2, 40, 4), (28, 31, 4), (29, 32, 6), (30, 33, 4), (58, 64, 4),
                                         (59, 65, 6), (40, 2, 4)])
@pytest.mark.parametrize("limiter", [0, 1])
@pytest.mark.parametrize("fp32", [False, True])
def test_two_iterations(nx, ny, order, limiter, fp32):
    import torch
    from paper_2507_03975_gb300 import gsis
    p = W.random_problem(nx, ny, order=order, seed=nx + 7 * ny)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    opt = gsis.default_options(scheme=gsis.SCHEME_SI, spatial_order=2, limiter=limiter, fixed_iters=2, max_iter=2,
                               precision=gsis.FP32_SWEEP if fp32 else gsis.FP64)
    r = gsis.solve(p.dx, p.dy, p.mu, p.eta, p.w, t(p.sigma_a), t(p.sigma_s), t(p.q), t(p.inflow.reshape(-1)), opt)
    o = oracle_uw2.solve(p, "si", fixed_iters=2, limiter="bj" if limiter == 0 else "none")
    err = np.abs(r["rho"].cpu().numpy() - o["rho"]).max() / np.abs(o["rho"]).max()
    assert err <= (1e-5 if fp32 else 1e-11), err


@pytest.mark.parametrize("exponent", [-460, 460])
def test_power_of_two_scaling_is_exact(exponent):
    """Intensities outside the exponents for which the limiter forms its ratio
    itself: scaling every source by a power of two scales every operation
    exactly, so the bits are those of the unscaled run."""
    import torch
    from paper_2507_03975_gb300 import gsis
    p = W.random_problem(37, 41, order=4, seed=11)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    opt = gsis.default_options(scheme=gsis.SCHEME_SI, spatial_order=2, limiter=0, fixed_iters=2, max_iter=2)
    rho = [gsis.solve(p.dx, p.dy, p.mu, p.eta, p.w, t(p.sigma_a), t(p.sigma_s), t(p.q * s),
                      t(p.inflow.reshape(-1) * s), opt)["rho"].cpu().numpy() / s for s in (1.0, 2.0 ** exponent)]
    assert np.array_equal(rho[0], rho[1])
