"""The reflections of a quadrature's directions (csrc/reflections.h, mom_quads)
against their definition, pair by pair, and in time that grows little faster
than the number of directions (4096 are accepted)."""
import time

import numpy as np
import pytest

import workloads as W
from test_moments_fixed_host import _p, lib  # noqa: F401


def _random(rng, kind):
    """Closed sets in any order, and what breaks them."""
    n = int(rng.integers(1, 40))
    mu, eta, w = rng.choice([0.1, 0.3, 0.5, 0.6], n) + 1e-3 * rng.integers(0, 3, n), rng.uniform(0.1, 0.7, n), rng.uniform(0.5, 1.0, n)
    mu, eta, w = np.concatenate([mu, -mu, mu, -mu]), np.concatenate([eta, eta, -eta, -eta]), np.concatenate([w] * 4)
    k = rng.integers(len(mu))
    if kind == "weight":
        w[k] *= 1.5
    elif kind == "sign":
        mu[k] = -mu[k]
    elif kind == "zero":
        eta[np.abs(eta) == abs(eta[k])] = 0.0
    elif kind == "twice":
        mu, eta, w = (np.concatenate([a, a[np.abs(eta) == abs(eta[k])]]) for a in (mu, eta, w))
    elif kind == "two weights":
        mu, eta, w = np.concatenate([mu] * 2), np.concatenate([eta] * 2), np.concatenate([w, 1.1 * w])
    order = rng.permutation(len(mu))
    return mu[order], eta[order], w[order]


def _quads(mu, eta, w):
    """Ascending quads of distinct directions with one weight, or None."""
    out = []
    for s in range(len(mu)):
        if mu[s] == 0 or eta[s] == 0:
            return None
        if mu[s] > 0 and eta[s] > 0:
            at = [np.flatnonzero((mu == a * mu[s]) & (eta == b * eta[s]) & (w == w[s])) for b in (1, -1) for a in (1, -1)]
            if any(len(t) != 1 for t in at):
                return None
            out.append([t[0] for t in at])
    return np.array(out) if 4 * len(out) == len(mu) else None


def _call(lib, mu, eta, w):
    K = len(mu)
    mu, eta, w = (np.ascontiguousarray(a) for a in (mu, eta, w))
    table, rep, nxt = np.zeros((K // 4 + 1, 16), np.uint32), np.empty(K, np.int32), np.empty(K, np.int32)
    n = lib.chains(K, _p(mu), _p(eta), _p(rep), _p(nxt))
    return lib.set_quads(K, _p(mu), _p(eta), _p(w), _p(table)), table, rep[:n], nxt


@pytest.mark.parametrize("kind", ["closed", "weight", "sign", "zero", "twice", "two weights"])
@pytest.mark.parametrize("seed", range(12))
def test_against_the_definition(lib, kind, seed):  # noqa: F811
    mu, eta, w = _random(np.random.default_rng(seed), kind)
    moments, table, rep, nxt = _call(lib, mu, eta, w)
    ref = _quads(mu, eta, w)
    assert (moments > 0) == (ref is not None)
    if ref is not None:
        assert np.array_equal(table[:len(ref), :4], ref)
    groups = {}
    for s, k in enumerate(zip(np.abs(mu), np.abs(eta))):
        groups.setdefault(k, []).append(s)
    assert sorted(g[0] for g in groups.values()) == list(rep)
    for g in groups.values():
        assert [nxt[s] for s in g] == g[1:] + [-1]


def test_time_grows_with_the_directions_not_with_their_pairs(lib):  # noqa: F811
    def best(K):
        """Closed sets without a common magnitude: every pair would be looked at."""
        rng = np.random.default_rng(K)
        mu, eta = rng.uniform(0.1, 0.7, K // 4), rng.uniform(0.1, 0.7, K // 4)
        s = (np.concatenate([mu, -mu, mu, -mu]), np.concatenate([eta, eta, -eta, -eta]), np.full(K, 4 * np.pi / K))
        t = []
        for _ in range(15):
            t0 = time.perf_counter()
            _call(lib, *s)
            t.append(time.perf_counter() - t0)
        return min(t)

    assert best(4096) < 9.0 * best(1024)   # 4.8 by the sort, 16 by pairs


@pytest.mark.parametrize("order", [4, 8, 16])
def test_level_symmetric_sets_are_quads(lib, order):  # noqa: F811
    mu, eta, w = W.level_symmetric_2d(order)
    moments, table, rep, _ = _call(lib, mu, eta, w)
    assert moments == 6 and np.array_equal(table[:len(mu) // 4, :4], _quads(mu, eta, w)) and len(rep) == len(mu) // 4
