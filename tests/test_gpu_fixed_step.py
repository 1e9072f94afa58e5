"""FP64 steps in fixed point against the FP64 arithmetic that runs where the positivity threshold is
not zero: the same lattices with a threshold of 1e-300, over the forms a handle accepts."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    from paper_2605_01774_gb300 import elbm
    elbm.lib()
    return elbm


def _start(dims, kind, seed):
    g = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*[np.arange(n) for n in dims[::-1]], indexing="ij")
    if kind == "smooth":
        return 1 + 0.3 * np.sin(2 * np.pi * x / dims[0]) * np.cos(2 * np.pi * (y / dims[1] + z / dims[2]))
    if kind == "plume":                                # far tails: the fallback, and nodes left to FP64
        return np.exp(-((x - dims[0] / 2) ** 2 + (y - dims[1] / 2) ** 2 + (z - dims[2] / 2) ** 2) / 6.0)
    if kind == "tiny":
        return 1e-290 * (1 + g.random(x.shape))
    return np.where(x < dims[0] // 2, 1.0, 0.0)         # "step": zeros beside ones


@pytest.mark.parametrize("kind", ["smooth", "plume", "tiny", "step"])
@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.06, -0.04, 0.02)])
@pytest.mark.parametrize("form", ["uniform", "field", "walls"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (7, 5, 3), (65, 9, 4), (40, 24, 18)])
def test_same_states(E, dims, form, u, kind):
    """8 steps.  Smooth states: a few FP64 roundings per step (2e-14 of the largest population), and
    the fallback at the same collisions.  Far tails and zeros beside ones, where the fallback and the
    stabilizer's guard multiply roundings: the 1e-12 that adversarial FP64 states are held to against
    the oracle."""
    phi0 = _start(dims, kind, 1)
    g = np.random.default_rng(2)
    n = int(np.prod(dims))
    states, counts = [], []
    if form != "uniform":
        q, _ = np.linalg.qr(g.standard_normal((n, 3, 3)))
        D = np.einsum("nij,nj,nkj->nik", q, 10.0 ** g.uniform(-4, -1, (n, 3)), q)
        D6 = np.ascontiguousarray(D[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]].T.astype(np.float32))
    for eps in (0.0, 1e-300):
        lat = E.Lattice(dims, "f64", bc=(1.2, 0.7) if form == "walls" and kind == "smooth" else None)
        if form == "uniform":
            E.elbm_set_tensor_uniform(lat.h, [0.05, 0.01, 0.0, 0.03, 0.005, 0.02])
        else:
            E.elbm_set_tensor_field(lat.h, D6)
            if form == "walls":
                E.elbm_set_source(lat.h, (1e-4 * np.random.default_rng(3).random(n) * phi0.max()).astype(np.float32))
        E.elbm_set_velocity_uniform(lat.h, u)
        E.elbm_set_params(lat.h, theta=1e-8, eps=eps)
        E.elbm_init_equilibrium(lat.h, phi0)
        E.elbm_step(lat.h, 8)
        out = np.empty((27, n))
        E.elbm_read_populations(lat.h, out)
        states.append(out)
        counts.append(E.elbm_reduce(lat.h, allow_nonfinite=True)["n_fallback"])
        lat.close()
    a, b = states
    assert np.isfinite(a).all()
    # the far tails of a plume and a step's zeros hang on thresholds that rounding decides
    if kind in ("smooth", "tiny"):
        assert counts[0] == counts[1]
    assert np.abs(a - b).max() <= (2e-14 if kind in ("smooth", "tiny") else 1e-12) * np.abs(b).max()


def test_non_finite_states_stay_visible(E):
    dims = (12, 8, 6)
    for bad in (np.nan, np.inf):
        phi0 = np.ones(dims[::-1])
        phi0[2, 3, 4] = bad
        lat = E.Lattice(dims, "f64")
        E.elbm_set_tensor_uniform(lat.h, [0.05, 0.01, 0.0, 0.03, 0.005, 0.02])
        E.elbm_set_velocity_uniform(lat.h, (0.05, 0.0, 0.0))
        E.elbm_init_equilibrium(lat.h, phi0)
        E.elbm_step(lat.h, 1)
        assert E.elbm_reduce(lat.h, allow_nonfinite=True)["status"] == 6
        lat.close()
