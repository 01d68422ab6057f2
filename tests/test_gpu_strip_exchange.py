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


@pytest.mark.parametrize("nx,ny", [(64, 64), (200, 200), (123, 123)])
def test_timeout_reports_and_next_call_recovers(nx, ny):
    """Waits bounded at 1 ns, less than any exchange takes: the call reports
    GSIS_ERR_DEVICE_TIMEOUT with all exchanges taken to their end, and the
    next call gives the oracle's answer (the solve ends at 1e-14 of the
    right-hand side; 1e-10 as for the other meshes)."""
    import oracle
    from paper_2507_03975_gb300 import gsis
    p = W.random_problem(nx, ny, order=4, seed=nx)
    sw = oracle.transport_sweep(p, np.random.default_rng(nx).uniform(0.0, 2.0, p.N))
    hx, hy = oracle.high_order_terms(p, sw["Fx"], sw["Fy"], *oracle.alsm_gradient(p, sw["rho"]))
    ref = oracle.SyntheticSolver(p).solve(oracle.synthetic_rhs(p, sw["rho"], hx, hy, sw["fb"]))
    args = (p.dx, p.dy, _t(p.sigma_a), _t(p.sigma_s), _t(p.q), _t(sw["rho"]),
            _t(np.concatenate([sw["Fx"], sw["Fy"]])), _t(sw["fb"]), None)
    for _ in range(20):
        with pytest.raises(gsis.GsisError) as e:
            gsis.synthetic_step(*args, gsis.default_options(synth_rtol=1e-14, synth_max_iter=3000, wait_limit_s=1e-9))
        assert e.value.status == gsis.GSIS_ERR_DEVICE_TIMEOUT
    r = gsis.synthetic_step(*args, gsis.default_options(synth_rtol=1e-14, synth_max_iter=3000))
    assert np.abs(r["rho"].cpu().numpy() - ref).max() < 1e-10 * np.abs(ref).max()
