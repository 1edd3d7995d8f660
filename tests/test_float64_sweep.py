"""The float64 sweep's functions return the values of the plain formulas bit for
bit (signs of zero aside): compiled for the host from the same source, on ordinary
states and where their short ways end (floors, zeros, jumps, supersonic and cold
flow, huge and tiny values, infinities, NaN)."""
import ctypes

import numpy as np
import pytest


@pytest.fixture(scope="module")
def hc():
    from paper_1810_01319_gb300 import build
    return ctypes.CDLL(build.build_hostcheck())


def _both(hc, what, x, out, gamma=5.0 / 3.0):
    x = np.ascontiguousarray(x, np.float64)
    fast, plain = np.zeros((len(x), out)), np.zeros((len(x), out))
    p = [ctypes.c_void_p(a.ctypes.data) for a in (x, fast, plain)]
    hc.cello_hc_q64(what, ctypes.c_long(len(x)), x.shape[1], p[0], ctypes.c_double(gamma), out, p[1], p[2])
    bad = ~((fast == plain) | (np.isnan(fast) & np.isnan(plain))).all(1)
    assert not bad.any(), (int(bad.sum()), x[bad][:3], fast[bad][:3], plain[bad][:3])


def _odd(rng, x, share=0.02):
    """Some values replaced by what no ordinary state holds."""
    special = np.array([0.0, -0.0, 1e-10, 1e-20, 1e-300, -1e-300, 5e-324, 1e160, -1e160, 1e300, np.inf, -np.inf,
                        np.nan, 1.0, -1.0])
    hit = rng.random(x.shape) < share
    x[hit] = rng.choice(special, int(hit.sum()))
    return x


def _primitives(rng, count, fields, kind):
    """States (rho, u, v, w, p[, e]): 0 smooth, 1 jumps, 2 supersonic, 3 cold, 4 at the floors, 5 at rest."""
    W = np.empty((count, fields))
    W[:, 0] = 10.0 ** rng.uniform(-1, 1, count) if kind else 1 + 0.1 * rng.standard_normal(count)
    W[:, 1:4] = rng.standard_normal((count, 3)) * (0.2, 1.0, 5.0, 3.0, 1.0, 0.0)[kind]
    W[:, 4] = 10.0 ** rng.uniform(-1, 1, count) if kind else 1 + 0.1 * rng.standard_normal(count)
    if kind == 3:
        W[:, 4] *= 1e-9
    if kind == 4:
        W[rng.random(count) < 0.5, 0] = 1e-10
        W[rng.random(count) < 0.5, 4] = 1e-20
    if fields == 6:
        W[:, 5] = W[:, 4] / W[:, 0] * 1.5
    return W


def test_quotients_and_roots(hc):
    rng = np.random.default_rng(1)
    n = 400000
    b = 2.0 ** rng.uniform(-119, 119, n)
    a = rng.choice([-1, 1], n) * 2.0 ** rng.uniform(-1000, 1000, n)
    a[::7] = b[::7] * rng.integers(1, 99, len(b[::7]))          # exact and nearly exact quotients
    a[::11] = np.nextafter(a[::11], 0)
    b[::13] = np.nextafter(2.0 ** rng.integers(-100, 100, len(b[::13])), 0)   # mantissas of ones
    _both(hc, 0, np.stack([a, b], 1), 1)
    _both(hc, 0, np.stack([_odd(rng, a, 0.5), b], 1), 1)
    x = 2.0 ** rng.uniform(-119, 119, n)
    k = rng.integers(1, 1 << 26, n).astype(float)
    x[::5] = (k * k)[::5]                                        # perfect squares and their neighbours
    x[::10] = np.nextafter(x[::10], 0)
    _both(hc, 1, x[:, None], 1)
    one = np.array([1 + k * 2.0 ** -52 for k in range(40)] + [1 - k * 2.0 ** -53 for k in range(1, 40)])
    ends = np.concatenate([one * s for s in (1.0, 0.5, 0.25, 2.0, 2.0 ** 40)])      # beside powers of two
    _both(hc, 1, ends[:, None], 1)
    c, d = np.meshgrid(ends, ends)
    _both(hc, 0, np.stack([c.ravel(), d.ravel()], 1), 1)


@pytest.mark.parametrize("kind", range(6))
@pytest.mark.parametrize("share", [0.0, 0.03])
def test_primitives_slopes_interfaces(hc, kind, share):
    rng = np.random.default_rng(10 + kind)
    n = 50000
    for fields, what in ((5, 2), (6, 12)):
        W = _primitives(rng, n, fields, kind)
        U = W.copy()
        U[:, 1:4] *= W[:, :1]
        U[:, 4] = W[:, 4] / (2 / 3) + 0.5 * W[:, 0] * (W[:, 1:4] ** 2).sum(1)
        if fields == 6:
            U[:, 5] *= W[:, 0]
        _both(hc, what, _odd(rng, U, share), fields)
    a = _primitives(rng, n, 5, kind)
    for q in range(5):
        x = np.stack([a[:, q], np.roll(a[:, q], 1), np.roll(a[:, q], 2), np.roll(a[:, q], 3)], 1)
        x[::9, 1] = x[::9, 0]
        x[::17, 1:] = np.nextafter(x[::17, :1], 9)
        x = _odd(rng, x, share)
        _both(hc, 3, x[:, :3], 1)
        _both(hc, 4, x, 1)
    x = np.concatenate([np.stack([np.roll(a[:, 4], i) for i in range(4)], 1), a[:, 1:2], np.roll(a[:, 1:2], 1, 0)], 1)
    x[:, 2] = np.where(rng.random(n) < 0.3, x[:, 1] * rng.uniform(1.2, 1.5, n), x[:, 2])
    x[::6, 3] = x[::6, 0]
    x[:, :4] = np.maximum(_odd(rng, x[:, :4].copy(), share), 1e-20)      # pressures come floored
    x[:, :4] = np.where(np.isnan(x[:, :4]), 1e-20, x[:, :4])
    x[:, 4:] = _odd(rng, x[:, 4:].copy(), share)
    _both(hc, 5, x, 1)


@pytest.mark.parametrize("kind", range(6))
@pytest.mark.parametrize("share", [0.0, 0.01])
@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.0005, 20.0])
def test_edge_states(hc, kind, share, gamma):
    rng = np.random.default_rng(30 + kind)
    n = 60000
    for fields, what in ((5, 6), (6, 16)):
        W = _primitives(rng, n, fields, kind)
        d = np.abs(W) * 0.2
        aL, aR = W + d * rng.standard_normal(W.shape), W + d * rng.standard_normal(W.shape)
        s = rng.random(W.shape)
        aL = np.where(s < 0.6, W - d * rng.random(W.shape), aL)          # monotone, some of them overshooting
        aR = np.where(s < 0.6, W + d * rng.random(W.shape) ** 3, aR)
        aL, aR = np.where(s > 0.9, W, aL), np.where(s > 0.95, W, aR)      # flat on one side or both
        f = np.where(rng.random((n, 1)) < 0.7, 0.0, np.where(rng.random((n, 1)) < 0.5, 1.0, rng.random((n, 1))))
        x = np.concatenate([_odd(rng, W, share), _odd(rng, aL, share), _odd(rng, aR, share), f,
                            np.full((n, 1), 0.05)], 1)
        W0, W4 = x[:, 0], x[:, 4]                                         # floored and never NaN
        x[:, 0], x[:, 4] = np.fmax(W0, 1e-10), np.fmax(W4, 1e-20)
        _both(hc, what, x, 2 * fields, gamma)


@pytest.mark.parametrize("kind", range(6))
@pytest.mark.parametrize("near", [0.0, 1e-12, 1e-6, 1e-3, 0.1, None])
@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.0005, 1.01, 20.0])
def test_two_shock_flux(hc, kind, near, gamma):
    rng = np.random.default_rng(50 + kind)
    n = 30000
    for fields, what in ((5, 7), (6, 17)):
        L = _primitives(rng, n, fields, kind)
        R = _primitives(rng, n, fields, kind) if near is None else L * (1 + near * rng.standard_normal(L.shape))
        if near is None:
            R[::3, 1] = L[::3, 1] + 20.0                                  # towards vacuum
            R[1::3, 1] = L[1::3, 1] - 20.0
            L, R = _odd(rng, L, 0.01), _odd(rng, R, 0.01)
        for S in (L, R):
            S[:, 0], S[:, 4] = np.fmax(S[:, 0], 1e-10), np.fmax(S[:, 4], 1e-20)
        _both(hc, what, np.concatenate([L, R], 1), fields + (fields == 6), gamma)
