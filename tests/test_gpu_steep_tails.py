"""FP64 plumes so narrow that their tails span hundreds of decades, and boxes that are empty around
them: node by node the fixed-point collision and FP64 arithmetic alternate there."""
import numpy as np
import pytest

import oracle as O
from test_fixed_collision import _collide, lib  # noqa: F401
from test_fixed_limits import _full, _run
from test_gpu_step_kernels import _staged_variants

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    from paper_2605_01774_gb300 import elbm
    elbm.lib()
    return elbm


def _bump(dims, width, cut=np.inf):
    z, y, x = np.meshgrid(*[np.arange(n) - (n - 1) / 2 for n in dims[::-1]], indexing="ij")
    r2 = x * x + y * y + z * z
    return np.where(r2 > cut * cut, 0.0, np.exp(-0.5 * r2 / width ** 2))


@pytest.mark.parametrize("u", [(0.05, 0.03, 0.02), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("width, cut", [(1.0, np.inf), (8.0, 8.0)])
def test_stays_finite(E, width, cut, u):
    """60 steps keep the mass to the 1e-12 that adversarial FP64 states are held to."""
    dims = (96, 80, 72)
    phi0 = _bump(dims, width, cut)
    lat = E.Lattice(dims, "f64")
    E.elbm_set_tensor_uniform(lat.h, [0.05, 0.01, 0.0, 0.03, 0.005, 0.02])
    E.elbm_set_velocity_uniform(lat.h, u)
    E.elbm_init_equilibrium(lat.h, phi0)
    E.elbm_step(lat.h, 60)
    d = E.elbm_reduce(lat.h, allow_nonfinite=True)
    lat.close()
    assert d["status"] == 0
    assert abs(d["mass"] - phi0.sum()) < 1e-12 * phi0.sum()


@pytest.mark.parametrize("walls", [None, (1.2, 0.7)])
@pytest.mark.parametrize("dims", [(1, 40, 30), (33, 7, 5), (64, 24, 18)])
def test_small_deciding_populations(E, lib, dims, walls):  # noqa: F811
    """One step, u = 0, from populations of which three in ten are 2 to 14 decades smaller than the
    others and decide the fallback of one node in a hundred, against the same header on the host.  Up to
    the FP32 quotients that remainders refine, both do the same integer arithmetic: what is left are 8
    units of the node (2^-57 of its largest 4^n g), times what the fallback makes of one, the largest
    4^n d over that of the deciding population."""
    n = int(np.prod(dims))
    g = np.random.default_rng(5)
    pops = O.W.numpy()[:, None] * g.uniform(0.3, 1.7, (27, n))
    pops = np.where(g.random((27, n)) < 0.3, pops * 10.0 ** g.uniform(-14, -2, (27, n)), pops)
    D6, still = [0.05, 0.01, 0.0, 0.03, 0.005, 0.02], np.zeros(3)
    lat = E.Lattice(dims, "f64", bc=walls)
    E.elbm_set_tensor_uniform(lat.h, D6)
    E.elbm_write_populations(lat.h, pops)
    E.elbm_read_populations(lat.h, pops)                 # wall nodes hold it to their rounding
    E.elbm_step(lat.h, 1)
    after = np.empty_like(pops)
    E.elbm_read_populations(lat.h, after)
    lat.close()
    T6 = np.ascontiguousarray(np.broadcast_to(np.asarray(E.elbm_relaxation_complement(D6)), (n, 6)))
    host, done, took = _run(lib, np.ascontiguousarray(pops.T), still, T6)
    assert done.mean() > 0.99 and took.sum() > 20
    scale = 4.0 ** (O.C.numpy() != 0).sum(1)[:, None]
    whole = _collide(pops, still, _full(T6), 1e-8, 0)[0]
    ratio = np.where(whole < 0, pops / np.where(whole < 0, pops - whole, 1), np.inf)
    d = np.abs(pops - whole) * scale
    grows = np.where(took, d.max(0) / d[ratio.argmin(0), np.arange(n)], 0.0)
    assert (grows > 16).sum() > (5 if n > 1000 else 0)
    unit = 2.0 ** (np.floor(np.log2((pops * scale).max(0))) - 57)
    most = 8 * (1 + grows) * unit / scale + 2.0 ** -52 * np.abs(host.T)
    at = np.arange(n).reshape(dims[::-1])
    for i, c in enumerate(O.C.numpy()):
        to = np.roll(at, (-c[2], -c[1], -c[0]), (0, 1, 2))      # the node that y sends population i to
        stays = done.reshape(at.shape).copy()
        if walls is not None and c[0] != 0:
            stays[:, :, -1 if c[0] > 0 else 0] = False
        y = at[stays]
        assert (np.abs(after[i, to[stays]] - host.T[i, y]) <= most[i, y]).all(), i


@pytest.mark.parametrize("u", [(0.05, 0.03, 0.02), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("dims", [(32, 11, 9), (96, 8, 5), (40, 12, 9), (48, 11, 7), (64, 9, 5)])
def test_step_kernels_agree(E, dims, u):
    """Which nodes are left to FP64 does not depend on the step kernel: bit-equal states after 12 steps of
    a plume two nodes wide, rows of whole warps and of 8 and 16 nodes more."""
    phi0 = _bump(dims, 2.0)
    states = []
    for variant in [1] + _staged_variants(E, dims, "f64", u=u):
        lat = E.Lattice(dims, "f64")
        E.elbm_set_tensor_uniform(lat.h, [0.05, 0.01, 0.0, 0.03, 0.005, 0.02])
        E.elbm_set_velocity_uniform(lat.h, u)
        E.elbm_set_step_kernel(lat.h, variant)
        E.elbm_init_equilibrium(lat.h, phi0)
        E.elbm_step(lat.h, 12)
        out = np.empty((27, phi0.size))
        E.elbm_read_populations(lat.h, out)
        states.append((out, E.elbm_reduce(lat.h)["n_fallback"]))
        lat.close()
    assert len(states) > 1
    for s, count in states[1:]:
        assert np.array_equal(s, states[0][0]) and count == states[0][1]
