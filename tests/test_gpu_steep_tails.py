"""FP64 plumes so narrow that their tails span hundreds of decades, and boxes that are empty around
them: node by node the fixed-point collision and FP64 arithmetic alternate there."""
import numpy as np
import pytest

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
