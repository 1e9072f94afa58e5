"""The fixed-point FP64 collision (csrc/fixed.cuh, compiled for the host) where its numbers reach the
ends of their range: at the onset of the positivity fallback, where it leaves a population at zero, where a
small population decides it, and at tensors that round to 2 and above."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
import torch
from test_fixed_collision import _collide, lib  # noqa: F401

THETA = 1e-8


def _tensors(g, n):
    q, _ = np.linalg.qr(g.standard_normal((n, 3, 3)))
    D = np.einsum("nij,nj,nkj->nik", q, 10.0 ** g.uniform(-6, -1, (n, 3)), q)
    T = 2 * np.eye(3) - np.linalg.inv(0.5 * np.eye(3) + 3 * D)
    return np.ascontiguousarray(T[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]])


def _full(T6):
    return T6[:, [[0, 1, 2], [1, 3, 4], [2, 4, 5]]]


def _equilibrium(u):
    return O.W.numpy() * O.eq_polynomial(torch.as_tensor(u)).numpy()


def _run(lib, pops, u, T6, fallback=1):  # noqa: F811
    """Collided nodes [n, 27], which were done in fixed point, and which took the fallback."""
    P, w, c = O.eq_polynomial(torch.as_tensor(u)).numpy(), O.W.numpy(), O.C.numpy()
    tables = np.concatenate([w * P, 3 * (1 / P - 1), np.log(P) - 3 * c @ u + 1.5 * u @ u, 1 / (w * P)])
    n = len(pops)
    out, flags, src = np.ascontiguousarray(pops.copy()), np.zeros(n, np.int32), np.zeros(n)
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    lib.run(C.c_long(n), p(out), p(np.ascontiguousarray(u)), p(tables), p(T6), p(src), 0, fallback, C.c_double(THETA),
            p(flags))
    return out, (flags & 1) == 1, (flags & 2) == 2


@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.05, 0.03, 0.02)])
def test_onset_of_the_fallback(lib, u):  # noqa: F811
    """Nodes bisected along a ray from the equilibrium to where some g* first turns negative, and a
    little beyond (1 - alpha from rounding size up to 2^-16): within the 1e-13 of the largest population
    that all nodes are held to, and none left to FP64 for its alpha."""
    u = np.array(u)
    g = np.random.default_rng(7)
    n = 4000
    E, T6 = _equilibrium(u), _tensors(g, n)
    ray = E * np.exp(1.0 * g.standard_normal((n, 27))) - E
    at = lambda s: E + s[:, None] * ray  # noqa: E731
    took = lambda s: _collide(at(s).T.astype(np.longdouble), u, _full(T6), THETA, 1)[1]  # noqa: E731
    ends = took(np.ones(n))
    assert ends.sum() > 200
    ray, T6, n = ray[ends], T6[ends], int(ends.sum())
    lo, hi = np.zeros(n), np.ones(n)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        t = took(mid)
        lo, hi = np.where(t, lo, mid), np.where(t, mid, hi)
    for beyond in (0.0, 2.0 ** -48, 2.0 ** -40, 2.0 ** -36, 2.0 ** -33, 2.0 ** -30, 2.0 ** -24, 2.0 ** -16):
        pops = at(hi * (1 + beyond))
        ref, fb = _collide(pops.T.astype(np.longdouble), u, _full(T6), THETA, 1)
        out, done, _ = _run(lib, pops, u, T6)
        err = (np.abs(out.T - ref).max(0) / np.abs(pops).max(1)).astype(float)
        assert done.mean() > 0.98, beyond
        assert err[done].max() < 1e-13, beyond


@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.05, 0.03, 0.02)])
def test_tensors_at_two(lib, u):  # noqa: F811
    """T < 2 for every finite D, but T of D = 1e15 rounds to 2 and above: the node is left to FP64, as
    are tensors that are not finite (uniform ones too); the largest T below 2 is taken, to 1e-13."""
    u = np.array(u)
    g = np.random.default_rng(11)
    E = _equilibrium(u)
    for bad in (2.0, np.nextafter(2.0, 3.0), -2.0, 4.0, 1e300, np.inf, np.nan):
        T6 = _tensors(g, 12)
        T6[np.arange(12), np.arange(12) // 2] = bad
        pops = E * (1 + 5e-3 * g.standard_normal((12, 27)))
        out, done, _ = _run(lib, pops, u, T6)
        assert not done[1::2].any(), bad                 # odd nodes have tensors of their own
        assert np.array_equal(out[1::2], pops[1::2])
        assert np.isfinite(bad) or not done[::2].any()
    T6 = _tensors(g, 6)
    T6[np.arange(6), [0, 0, 3, 3, 5, 5]] = np.nextafter(2.0, 0.0)
    pops = E * (1 + 5e-3 * g.standard_normal((6, 27)))
    ref, _ = _collide(pops.T.astype(np.longdouble), u, _full(T6), THETA, 1)
    out, done, _ = _run(lib, pops, u, T6)
    assert done.all()
    assert (np.abs(out.T - ref).max(0) / pops.max(1)).max() < 1e-13


@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.05, 0.03, 0.02)])
def test_fallback_leaves_nothing_negative(lib, u):  # noqa: F811
    """Populations that are not negative stay so, exactly: the fallback's deciding one becomes 0."""
    u = np.array(u)
    g = np.random.default_rng(13)
    n = 4000
    pops, T6 = _equilibrium(u) * np.exp(1.0 * g.standard_normal((n, 27))), _tensors(g, n)
    out, done, took = _run(lib, pops, u, T6)
    assert (done & took).sum() > 200
    assert out[done].min() >= 0.0


@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.05, 0.03, 0.02)])
@pytest.mark.parametrize("spread", [2.0, 4.0, 8.0])
def test_small_deciding_populations(lib, spread, u):  # noqa: F811
    """Populations that differ by decades, of which a small one often decides the fallback: no further
    from the exact collision than FP64 arithmetic is (root mean square over the nodes, relative to the
    largest population)."""
    u = np.array(u)
    g = np.random.default_rng(17)
    n = 40000
    pops, T6 = _equilibrium(u) * np.exp(spread * g.standard_normal((n, 27))), _tensors(g, n)
    out, done, took = _run(lib, pops, u, T6)
    assert (done & took).sum() > 1000
    pops, T6, out = pops[done], T6[done], out[done]
    ref, fb = _collide(pops.T.astype(np.longdouble), u, _full(T6), THETA, 1)
    assert np.array_equal(fb, took[done])
    f64 = _collide(pops.T, u, _full(T6), THETA, 1)[0]
    rms = lambda x: float(np.sqrt(((np.abs(x - ref).max(0) / pops.max(1)) ** 2).mean()))  # noqa: E731
    assert rms(out.T) <= rms(f64), (rms(out.T), rms(f64))
