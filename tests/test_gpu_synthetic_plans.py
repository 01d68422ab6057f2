"""The synthetic solvers where their plans change: strips cut at level 1 or
deeper, levels whose rows do not divide among the CTAs of a cluster (29, 61,
123), levels of at most 32 and of more than 1024 cells in one CTA, long thin
meshes either way, and the tiled solver's odd sub-tiles.

Tolerance: the solve ends at a residual of 1e-14 of the right-hand side, and
the diagonally dominant operators of these media have condition numbers below
1e4: 1e-10 of the largest value is asked, as of the other meshes.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 16), (29, 29), (31, 33), (61, 61), (64, 64), (123, 123), (18, 140), (5, 300),
                                   (300, 5), (33, 500), (200, 200), (245, 245), (331, 287)])
def test_against_direct_solve(nx, ny):
    import torch
    from paper_2507_03975_gb300 import gsis
    p = W.random_problem(nx, ny, order=4, seed=nx + 3 * ny)
    rng = np.random.Generator(np.random.PCG64(nx * ny))
    sw = oracle.transport_sweep(p, rng.uniform(0.0, 2.0, p.N))
    hx, hy = oracle.high_order_terms(p, sw["Fx"], sw["Fy"], *oracle.alsm_gradient(p, sw["rho"]))
    ref = oracle.SyntheticSolver(p).solve(oracle.synthetic_rhs(p, sw["rho"], hx, hy, sw["fb"]))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    opt = gsis.default_options(synth_rtol=1e-14, synth_max_iter=3000)
    r = gsis.synthetic_step(p.dx, p.dy, t(p.sigma_a), t(p.sigma_s), t(p.q), t(sw["rho"]),
                            t(np.concatenate([sw["Fx"], sw["Fy"]])), t(sw["fb"]), None, opt)
    err = np.abs(r["rho"].cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err < 1e-10, err
