"""The fixed-point moments (csrc/moments_fixed.cuh) compiled for the host,
against exact sums and the FP64 loop that they stand in for.

What is asked, of every moment and kind of cell: relative to the sum of the
terms' magnitudes, neither the largest nor the root-mean-square error over
the cells is larger than the loop's.  The exact sums are taken in long double
(64 bits of mantissa or more: their own error is below 1e-17).
"""
import ctypes
import subprocess
from pathlib import Path

import numpy as np
import pytest

import workloads as W

HERE = Path(__file__).resolve().parent
CELLS = 2000


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = tmp_path_factory.mktemp("moments") / "moments.so"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-w", "-fPIC", "-shared", "-ffp-contract=off",
                           "-I" + str(HERE.parent / "paper_2507_03975_gb300" / "csrc"),
                           str(HERE / "moments_fixed_host.cpp"), "-o", str(so)])
    return ctypes.CDLL(str(so))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _quads(mu, eta):
    """[K/4, 4]: the reflections (mu, eta), (-mu, eta), (mu, -eta), (-mu, -eta)."""
    at = {(m, e): k for k, (m, e) in enumerate(zip(mu, eta))}
    return np.array([[at[m, e], at[-m, e], at[m, -e], at[-m, -e]] for m, e in zip(mu, eta) if m > 0 and e > 0], np.int32)


def _table(mu, eta, w):
    q = _quads(mu, eta)
    k = q[:, 0]
    cf = np.stack([w[k], w[k] * mu[k], w[k] * eta[k], w[k] * mu[k] * mu[k], w[k] * mu[k] * eta[k], w[k] * eta[k] * eta[k]], 1)
    c = np.rint(np.ldexp(cf, 62)).astype(np.uint64)
    t = np.zeros((len(q), 16), np.uint32)
    t[:, :4] = q
    t[:, 4::2] = c >> np.uint64(32)
    t[:, 5::2] = c & np.uint64(0xffffffff)
    return np.ascontiguousarray(t)


def _intensities(kind, q, rng):
    K, n = q.size, CELLS
    if kind == "dense":
        return rng.uniform(0.5, 1.5, (K, n))
    if kind == "decades":
        return 10.0 ** rng.uniform(-20.0, 0.0, (K, n))
    if kind == "signed":
        return rng.normal(size=(K, n))
    if kind == "rising":   # in the order of the sum: every chunk holds a larger exponent
        I = np.empty((K, n))
        I[q.reshape(-1)] = np.sort(10.0 ** rng.uniform(-3.0, 0.0, (K, n)), 0)
        return I
    I = rng.uniform(0.5, 1.0, (K, n)) * 10.0 ** rng.uniform(-12.0, 0.0, (1, n))   # one strong ordinate
    I[rng.integers(K, size=n), np.arange(n)] = rng.uniform(1.0, 2.0, n)
    return I


def _errors(lib, mu, eta, w, table, I):
    """{number of moments: [cells, that many]} errors of the fixed-point sums, and the loop's [cells, 6]."""
    K, n = I.shape
    I = np.ascontiguousarray(I)
    ld = np.longdouble
    coef = np.ascontiguousarray([w, w * mu, w * eta, w * mu * mu, w * mu * eta, w * eta * eta])
    m, e = mu.astype(ld), eta.astype(ld)
    terms = [(w.astype(ld) * f)[:, None] * I.astype(ld) for f in (ld(1), m, e, m * m, m * e, e * e)]
    exact = np.stack([t.sum(0) for t in terms], 1)
    size = np.stack([np.abs(t).sum(0) for t in terms], 1)
    loop = np.empty((n, 6))
    lib.loop_cells(K, _p(coef), _p(I), n, _p(loop))
    fixed = {}
    for nm in (1, 3, 6):
        out, ok = np.empty((n, nm)), np.zeros(n, np.uint8)
        lib.fixed_cells(nm, _p(table), len(table), _p(I), n, _p(out), _p(ok))
        assert ok.all()
        fixed[nm] = (np.abs(out.astype(ld) - exact[:, :nm]) / size[:, :nm]).astype(float)
    return fixed, (np.abs(loop.astype(ld) - exact) / size).astype(float)


@pytest.mark.parametrize("kind", ["dense", "decades", "signed", "rising", "beam"])
@pytest.mark.parametrize("order", [4, 6, 8, 10, 12, 14, 16])
def test_level_symmetric_no_worse_than_the_loop(lib, order, kind):
    mu, eta, w = W.level_symmetric_2d(order)
    I = _intensities(kind, _quads(mu, eta), np.random.default_rng(order))
    fixed, loop = _errors(lib, mu, eta, w, _table(mu, eta, w), I)
    for nm, f in fixed.items():
        for m in range(nm):
            assert f[:, m].max() <= loop[:, m].max(), (nm, m)
            assert np.sqrt((f[:, m] ** 2).mean()) <= np.sqrt((loop[:, m] ** 2).mean()), (nm, m)


def _product(azimuthal, polar):
    """Gauss-Legendre levels x equally spaced angles per quadrant; the smallest w mu^2 gets very small."""
    x, wx = np.polynomial.legendre.leggauss(2 * polar)
    x, wx = x[polar:], wx[polar:]
    phi = (np.arange(azimuthal) + 0.5) * np.pi / 2 / azimuthal
    s = np.sqrt(1.0 - x * x)[:, None]
    mu, eta = (s * np.cos(phi)).reshape(-1), (s * np.sin(phi)).reshape(-1)
    w = np.repeat(wx, azimuthal)
    return _all_quadrants(mu, eta, w * (np.pi / w.sum()))


def _all_quadrants(mu, eta, w):
    return (np.concatenate([mu, -mu, mu, -mu]), np.concatenate([eta, eta, -eta, -eta]), np.concatenate([w] * 4))


def _small_weight(wt):
    """S8 with one direction (and its reflections) of weight wt."""
    mu, eta, w = W.level_symmetric_2d(8)
    w = w.copy()
    small = (np.abs(mu) == abs(mu[3])) & (np.abs(eta) == abs(eta[3]))
    w[small] = wt
    w[~small] *= (4.0 * np.pi - wt * small.sum()) / w[~small].sum()
    return mu, eta, w


SETS = {**{f"S{o}": W.level_symmetric_2d(o) for o in (4, 8, 16)},
        **{f"product {a}x{p}": _product(a, p) for a, p in ((2, 1), (4, 2), (6, 3), (8, 4), (16, 16))},
        **{f"weight {wt:g}": _small_weight(wt) for wt in (1e-2, 1e-6, 1e-9, 1e-15, 1e-20)}}


@pytest.mark.parametrize("name", SETS)
def test_no_set_is_worse_than_the_loop(lib, name):
    """Of the moments that mom_quads lets through, and with the strong ordinate
    in each direction in turn, the smallest coefficients among them."""
    mu, eta, w = SETS[name]
    K = len(mu)
    table = np.zeros((K // 4, 16), np.uint32)
    nm = lib.set_quads(K, _p(np.ascontiguousarray(mu)), _p(np.ascontiguousarray(eta)), _p(np.ascontiguousarray(w)), _p(table))
    assert nm in (0, 3, 6)
    assert nm == 6 if name[0] == "S" else nm == 0 if w.min() < 1e-4 else True
    if nm == 0:
        return
    rng = np.random.default_rng(K)
    for kind in ("dense", "decades", "signed", "rising", "beam"):
        I = _intensities(kind, _quads(mu, eta), rng)
        if kind == "beam":   # all directions alike
            I[:] = rng.uniform(0.5, 1.0, I.shape) * 10.0 ** rng.uniform(-12.0, -2.0, (1, CELLS))
            I[np.arange(CELLS) % K, np.arange(CELLS)] = rng.uniform(1.0, 2.0, CELLS)
        fixed, loop = _errors(lib, mu, eta, w, table, I)
        for n in (1, 3, 6)[:{3: 2, 6: 3}[nm]]:
            for m in range(n):
                assert fixed[n][:, m].max() <= loop[:, m].max(), (kind, n, m)
                assert np.sqrt((fixed[n][:, m] ** 2).mean()) <= np.sqrt((loop[:, m] ** 2).mean()), (kind, n, m)


@pytest.mark.parametrize("value", [2.0 - 2.0 ** -52, -(2.0 - 2.0 ** -52)])
@pytest.mark.parametrize("name", SETS)
def test_largest_sums_fit(lib, name, value):
    """All mantissas full: the sums reach their largest magnitudes."""
    mu, eta, w = SETS[name]
    K = len(mu)
    table = np.zeros((K // 4, 16), np.uint32)
    nm = lib.set_quads(K, _p(np.ascontiguousarray(mu)), _p(np.ascontiguousarray(eta)), _p(np.ascontiguousarray(w)), _p(table))
    for n in (3, 6):
        if n > nm:
            continue
        I, out, ok = np.full((K, 1), value), np.empty((1, n)), np.zeros(1, np.uint8)
        lib.fixed_cells(n, _p(table), K // 4, _p(I), 1, _p(out), _p(ok))
        ref = np.array([(w * f).sum() * value for f in (1.0, 0 * mu, 0 * eta, mu * mu, 0 * mu, eta * eta)])[:n]
        assert ok[0] and np.abs(out[0] - ref).max() < 1e-14 * abs(ref[0])
