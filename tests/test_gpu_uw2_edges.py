"""The second-order residual kernel at its strips' real height (16 rows, the
row before the first formed again) and with a number of ordinates that does
not fill its blocks of four warps, with and without the limiter.

Tolerance: as for the strips' width (test_gpu_uw2_strips.py): the operations
are the oracle's up to the order of a few roundings, which two iterations
amplify by less than 1e4: 1e-11 of the largest value (FP32: 1e-5).
"""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import uw2 as oracle_uw2

pytestmark = pytest.mark.gpu


def _directions(K, rng):
    r, a = np.sqrt(rng.uniform(0.05, 0.95, K)), rng.uniform(0.0, 2.0 * np.pi, K)
    w = rng.uniform(0.5, 1.5, K)
    return r * np.cos(a), r * np.sin(a), w * (4.0 * np.pi / w.sum())


@pytest.mark.parametrize("nx,ny,K", [(30, 15, 4), (29, 16, 5), (31, 17, 6), (12, 31, 7), (59, 32, 9), (33, 33, 1),
                                     (20, 48, 13), (3, 49, 2)])
@pytest.mark.parametrize("limiter", [0, 1])
@pytest.mark.parametrize("fp32", [False, True])
def test_two_iterations(nx, ny, K, limiter, fp32):
    import torch
    from paper_2507_03975_gb300 import gsis
    rng = np.random.default_rng(100 * nx + ny)
    mu, eta, w = _directions(K, rng)
    base = W.random_problem(nx, ny, order=4, seed=nx + 7 * ny)
    p = dataclasses.replace(base, mu=mu, eta=eta, w=w, inflow=rng.uniform(0.0, 1.0, (base.n_bface, K)))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    opt = gsis.default_options(scheme=gsis.SCHEME_SI, spatial_order=2, limiter=limiter, fixed_iters=2, max_iter=2,
                               precision=gsis.FP32_SWEEP if fp32 else gsis.FP64)
    r = gsis.solve(p.dx, p.dy, p.mu, p.eta, p.w, t(p.sigma_a), t(p.sigma_s), t(p.q), t(p.inflow.reshape(-1)), opt)
    o = oracle_uw2.solve(p, "si", fixed_iters=2, limiter="bj" if limiter == 0 else "none")
    err = np.abs(r["rho"].cpu().numpy() - o["rho"]).max() / np.abs(o["rho"]).max()
    assert err <= (1e-5 if fp32 else 1e-11), err
