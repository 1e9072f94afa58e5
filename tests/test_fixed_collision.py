"""The fixed-point FP64 collision (csrc/fixed.cuh) compiled for the host, node by node against the
collision in extended precision (itself held to the FP64 oracle where that is well conditioned):
every form it accepts, at every distance from equilibrium."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_01774_gb300", "csrc")
HARNESS = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "fixed.cuh"
using namespace elbm;
struct K { double E[Q], K3[Q], L[Q], M[Q], ux, uy, uz, theta2, eps; Sym6<double> T; };
// nodes [n][27] in place; T [n][6]; src [n]; out flags: 1 done in fixed point, 2 fallback taken
extern "C" void run(long n, double* g, const double* u, const double* tables, const double* T, const double* src,
                    int has_src, int fallback, double theta, int* flags) {
  K k;
  for (int i = 0; i < Q; ++i) { k.E[i] = tables[i]; k.K3[i] = tables[27 + i]; k.L[i] = tables[54 + i]; k.M[i] = tables[81 + i]; }
  k.ux = u[0]; k.uy = u[1]; k.uz = u[2]; k.theta2 = theta * theta; k.eps = 0;
  for (long m = 0; m < n; ++m) {
    const double* t = T + 6 * m;
    k.T = Sym6<double>{t[0], t[1], t[2], t[3], t[4], t[5]};
    const FixConsts f = fix_consts(k);
    bool took = false;
    InLocal keep;
    double v[Q];
    for (int i = 0; i < Q; ++i) v[i] = g[27 * m + i];
    auto out = [&](int i, double x) { g[27 * m + i] = x; };
    const double* tn = m % 2 ? t : nullptr;          // the node's own tensor, or the uniform one
    const bool still = u[0] == 0 && u[1] == 0 && u[2] == 0;
    const bool done = f.ok && (still ? collide_fixed<0>(v, tn, src[m], has_src, fallback, f, keep, took, out)
                                     : collide_fixed<1>(v, tn, src[m], has_src, fallback, f, keep, took, out));
    flags[m] = (done ? 1 : 0) | (took ? 2 : 0);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "h.cpp").write_text(HARNESS)
    so = d / "h.so"
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(d / "h.cpp")], check=True)
    return C.CDLL(str(so))


def _nodes(u, spread, scale, seed, n=400):
    g = np.random.default_rng(seed)
    P = O.eq_polynomial(torch.as_tensor(u)).numpy()
    E = O.W.numpy() * P
    noise = g.standard_normal((n, 27))
    pops = E * (np.exp(spread * noise) if spread > 0.5 else 1 + spread * noise) * scale
    d = 10.0 ** g.uniform(-6, -1, (n, 3))
    q, _ = np.linalg.qr(g.standard_normal((n, 3, 3)))
    D = np.einsum("nij,nj,nkj->nik", q, d, q)
    src = scale * 1e-3 * g.standard_normal(n)
    return pops, D, src, P


def _collide(g, u, T, theta, fallback):
    """Section 2.7's collision of g [27, n] with T = 2I - S [n, 3, 3], in g's precision."""
    w, c = O.W.numpy().astype(g.dtype), O.C.numpy().astype(g.dtype)
    n = (O.C.numpy() != 0).sum(1)
    w = np.array([8, 2, 0, 0], g.dtype)[np.minimum(n, 1)] / 27
    w[n == 2], w[n == 3] = g.dtype.type(1) / 54, g.dtype.type(1) / 216
    u = u.astype(g.dtype)
    cu = c @ u
    P = 1 + 3 * cu + g.dtype.type(4.5) * cu * cu - g.dtype.type(1.5) * (u @ u)
    phi = g.sum(0)
    j = c.T @ g - u[:, None] * phi
    a = np.einsum("nij,jn->in", T.astype(g.dtype), j) - j
    dh = g - (w * P)[:, None] * phi - 3 * w[:, None] * (c @ j)
    out = (w * P)[:, None] * phi + 3 * w[:, None] * (c @ a)
    if (u != 0).any():
        num = (dh * ((3 * (1 / P - 1))[:, None] * (c @ a) / phi + (np.log(P) - 3 * cu + g.dtype.type(1.5) * (u @ u))[:, None])).sum(0)
        den = (dh * dh / (w * P)[:, None]).sum(0) / phi
        on = den > g.dtype.type(theta) ** 2 * phi
        out = out - np.where(on, num / np.where(on, den, 1), 0) * dh
    took = np.zeros(g.shape[1], bool)
    if fallback:
        took = (out < 0).any(0)
        om = out - g
        r = np.where(om < 0, g / np.where(om < 0, -om, 1), np.inf).min(0).clip(0, 1)
        out = np.where(took, g + r * om, out)
    return out, took


@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.05, 0.03, 0.02), (-0.12, 0.0, 0.09)])
@pytest.mark.parametrize("spread", [1e-7, 1e-3, 0.1, 0.3, 1.0])
@pytest.mark.parametrize("fallback,has_src,scale", [(1, 0, 1.0), (0, 1, 1.0), (1, 1, 1e-200), (1, 0, 1e150)])
def test_against_extended_precision(lib, u, spread, fallback, has_src, scale):
    """Within 1e-13 of the node's largest population (a few hundred FP64 roundings), and no further
    from the exact collision than FP64 arithmetic is."""
    u = np.array(u)
    pops, D, src, P = _nodes(u, spread, scale, 3)
    n = len(pops)
    T = 2 * np.eye(3) - np.linalg.inv(0.5 * np.eye(3) + 3 * D)
    T6 = np.ascontiguousarray(T[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]])
    w, c = O.W.numpy(), O.C.numpy()
    tables = np.concatenate([w * P, 3 * (1 / P - 1), np.log(P) - 3 * c @ u + 1.5 * u @ u, 1 / (w * P)])
    out, flags = np.ascontiguousarray(pops.copy()), np.zeros(n, dtype=np.int32)
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    lib.run(C.c_long(n), p(out), p(np.ascontiguousarray(u)), p(tables), p(T6), p(src), has_src, fallback,
            C.c_double(1e-8), p(flags))
    done = (flags & 1) == 1
    assert done.mean() > (0.95 if spread < 0.5 else 0.8)
    g = pops.T.astype(np.longdouble)
    if has_src:
        g = g + src.astype(np.longdouble) * (w * P).astype(np.longdouble)[:, None]
    T = T6[:, [[0, 1, 2], [1, 3, 4], [2, 4, 5]]]
    ref, took = _collide(g, u, T, 1e-8, fallback)
    size = np.abs(g).max(0)
    err = (np.abs(out.T - ref).max(0) / size).astype(float)
    f64 = _collide((g / scale).astype(np.float64), u, T, 1e-8, fallback)[0]
    f64 = (np.abs(f64 - ref / scale).max(0) / (size / scale)).astype(float)
    ok = done
    if spread < 1e-6:
        # kappa dh is a quotient of residues of 1e-7 phi: FP64 itself is 1e-12 to 1e-11 off, and
        # rounding decides which nodes cross the stabilizer's guard
        ok = done & (f64 < 1e-9) & (err < 1e-9)
        assert ok.mean() > 0.95
    else:
        assert err[done].max() < 1e-13
    if spread < 0.5:
        assert np.sqrt((err[ok] ** 2).mean()) <= np.sqrt((f64[ok] ** 2).mean())
    assert np.array_equal((flags[done] & 2) == 2, took[done])
    if spread > 1e-6:
        S = torch.as_tensor(2 * np.eye(3) - T)
        o, info = O.collide(torch.as_tensor((g / scale).astype(np.float64)), torch.as_tensor(u), S, theta=1e-8,
                            lam_mode="reduced", fallback=bool(fallback))
        assert np.array_equal(info.fallback.numpy(), took)
        assert (np.abs(o.numpy() - ref / scale).max(0) / np.abs(g / scale).max(0)).max() < 1e-13


def test_refuses_what_it_cannot_hold(lib):
    u = np.array([0.05, 0.0, 0.0])
    pops, D, src, P = _nodes(u, 1e-3, 1.0, 5, n=6)
    pops[0, 4], pops[1, 9], pops[2] = np.inf, np.nan, 0.0
    pops[3] *= 1e-300
    pops[4] = -pops[4]
    w, c = O.W.numpy(), O.C.numpy()
    tables = np.concatenate([w * P, 3 * (1 / P - 1), np.log(P) - 3 * c @ u + 1.5 * u @ u, 1 / (w * P)])
    T6 = np.ascontiguousarray(np.tile([0.3, 0, 0, 0.3, 0, 0.3], (6, 1)))
    out, flags = pops.copy(), np.zeros(6, dtype=np.int32)
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    lib.run(C.c_long(6), p(out), p(u), p(tables), p(T6), p(src), 0, 1, C.c_double(1e-8), p(flags))
    assert list(flags & 1) == [0, 0, 0, 0, 0, 1]
    assert np.array_equal(out[:5], pops[:5], equal_nan=True)
