"""Moments of the kinetic step for quadratures other than level-symmetric
ones: product sets, whose w mu^2 get small, and sets with one very small
weight, whose ordinate carries a beam of intensity 1 / w.

Every term is positive (sources, inflow and coefficients of rho, P_xx, P_yy),
so each cell's value is asked to a relative 1e-13: a chain of at most nx + ny
cells and sums of K <= 128 terms round to less than (nx + ny + K) 2^-53 of it.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads as W
from test_moments_fixed_host import _product, _small_weight

pytestmark = pytest.mark.gpu

SETS = {"product 4x2": _product(4, 2), "product 8x4": _product(8, 4),
        **{f"weight {wt:g}": _small_weight(wt) for wt in (1e-2, 1e-6, 1e-9, 1e-15, 1e-20)}}


@pytest.mark.parametrize("name", SETS)
@pytest.mark.parametrize("quadrant", [0, 3])
def test_beam_in_the_direction_of_the_smallest_coefficient(name, quadrant):
    import torch
    from paper_2507_03975_gb300 import gsis
    mu, eta, w = SETS[name]
    K = len(mu)
    base = W.random_problem(21, 26, order=4, seed=K)
    k = int(np.argmin((w * mu * mu)[:K // 4])) + quadrant * K // 4
    inflow = np.full((base.n_bface, K), 1e-4)
    inflow[:, k] = 1.0 / w[k]
    p = dataclasses.replace(base, mu=mu, eta=eta, w=w, inflow=inflow)
    rho = np.random.default_rng(K).uniform(0.0, 1e-3, p.N)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    r = gsis.transport_sweep(p.dx, p.dy, p.mu, p.eta, p.w, t(p.sigma_a), t(p.sigma_s), t(p.q), t(rho),
                             t(inflow.reshape(-1)))
    o = oracle.transport_sweep(p, rho)
    P = r["P"].cpu().numpy().reshape(3, -1)
    for name, a, b in (("rho", r["rho"].cpu().numpy(), o["rho"]), ("Pxx", P[0], o["Pxx"]), ("Pyy", P[2], o["Pyy"])):
        assert (np.abs(a / b - 1.0) <= 1e-13).all(), (name, np.abs(a / b - 1.0).max())
