"""Fixed-point angular moments of FP64 intensities (csrc/moments_fixed.cuh)
against the oracle's plain FP64 sums: numbers of quads that fill no whole
chunk, one to a few cells, negative and zero intensities, a single beam, and
scales from the smallest normal numbers (where the kernel takes its plain
loop) to large ones.

Tolerance: the kinetic step and both sums round to 2^-53 a term; over a chain
of at most nx + ny cells and K terms of one magnitude that is below
(nx + ny + K) 2^-53 < 4e-14 of the largest value; 1e-13 is asked.  Scaling
every source by a power of two is exact, down to the spacing 2^-1074 of the
smallest numbers.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _sweep(p, rho, scale=1.0):
    from paper_2507_03975_gb300 import gsis
    inflow = None if p.inflow is None else _t(p.inflow.reshape(-1) * scale)
    r = gsis.transport_sweep(p.dx, p.dy, p.mu, p.eta, p.w, _t(p.sigma_a), _t(p.sigma_s), _t(p.q * scale),
                             _t(rho * scale), inflow)
    return {k: r[k].cpu().numpy() for k in ("rho", "F", "P")}


def _check(p, rho, scale=1.0):
    r = _sweep(p, rho, scale)
    o = oracle.transport_sweep(p, rho)
    ref = {"rho": o["rho"], "F": np.concatenate([o["Fx"], o["Fy"]]),
           "P": np.concatenate([o["Pxx"], o["Pxy"], o["Pyy"]])}
    big = np.abs(o["rho"]).max()
    for k, v in ref.items():
        err = np.abs(r[k] / scale - v).max()
        assert err <= 1e-13 * big + p.K * 2.0 ** -1074 / scale, (k, err, big)


@pytest.mark.parametrize("nx,ny,order", [(1, 1, 4), (3, 2, 6), (33, 5, 8), (17, 40, 10), (64, 31, 12), (20, 33, 16)])
def test_matches_oracle(nx, ny, order):
    p = W.random_problem(nx, ny, order=order, seed=nx + order)
    _check(p, np.random.default_rng(order).uniform(0.0, 2.0, p.N))


@pytest.mark.parametrize("exponent", [-1040, -1000, -960, -900, 0, 900])
def test_scales(exponent):
    p = W.random_problem(19, 23, order=8, seed=5)
    _check(p, np.random.default_rng(6).uniform(0.0, 2.0, p.N), 2.0 ** exponent)


def test_signs_and_zeros():
    p = W.random_problem(21, 18, order=8, seed=8)
    q = np.random.default_rng(9).normal(0.0, 1.0, p.N)
    p = dataclasses.replace(p, q=q, inflow=p.inflow - 0.5)
    _check(p, np.zeros(p.N))
    z = dataclasses.replace(p, q=np.zeros(p.N), inflow=None)
    assert all(not v.any() for v in _sweep(z, np.zeros(p.N)).values())


@pytest.mark.parametrize("k", [0, 5, 17, 33])
def test_single_beam(k):
    p = W.homogeneous(24, 20, order=8, sigma_t=3.0, ratio=0.0, q=0.0)
    inflow = np.zeros((p.n_bface, p.K))
    inflow[:, k] = 1.0
    _check(dataclasses.replace(p, inflow=inflow), np.zeros(p.N))
