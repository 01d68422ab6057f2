"""The strip synthetic solver's exchanges between the CTAs of a cluster
(csrc/mg.cu, SCluster)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("nx,ny,count", [(64, 64, 96), (48, 130, 40)])
def test_crowded_batch_equals_single_solve(nx, ny, count):
    """Many clusters at once, several CTAs to an SM, so that the CTAs of one
    cluster start and load at different speeds.  With two inner iterations
    the solve does not correct a value that a neighbour's late clearing would
    have lost, so every problem must end with the single solve's bits."""
    from paper_2507_03975_gb300 import gsis
    p = W.random_problem(nx, ny, order=4, seed=nx + ny)
    d = dict(dx=p.dx, dy=p.dy, mu=p.mu, eta=p.eta, w=p.w, sigma_a=_t(p.sigma_a), sigma_s=_t(p.sigma_s), q=_t(p.q),
             inflow=_t(p.inflow.reshape(-1)))
    opt = gsis.default_options(fixed_iters=4, max_iter=4, synth_max_iter=2, beta=10.0)
    one = gsis.solve(*[d[k] for k in ("dx", "dy", "mu", "eta", "w", "sigma_a", "sigma_s", "q", "inflow")], opt,
                     want_P=False)["rho"].cpu().numpy()
    for _ in range(5):
        tuning = gsis.default_batch_tuning(synth_cells_per_cta=0)   # the single solve's cluster size
        r = gsis.solve_batch([d] * count, opt, tuning=tuning)["results"]
        assert all(np.array_equal(x["rho"].cpu().numpy(), one) for x in r)
