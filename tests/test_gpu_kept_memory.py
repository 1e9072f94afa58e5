"""Device memory that handles keep for speed: what is taken by default, what the caller's limits give
back, and the same bits either way."""
import pytest
import torch

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def E():
    from paper_2605_01774_gb300 import elbm
    elbm.lib()
    return elbm


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_velocity_tables(E):
    """700 x 600 FP64 nodes: 121 MB of tables.  None with a limit of 0, set before the field or after it
    (while steps run), and the states are those with the tables kept."""
    nx, ny = 700, 600
    tables = 288 * nx * ny
    gen = torch.Generator(device="cuda").manual_seed(2)
    phi = 0.5 + torch.rand((ny, nx), generator=gen, device="cuda")
    u = 0.2 * torch.rand((2, ny, nx), generator=gen, device="cuda") - 0.1
    states = []
    for when in ("kept", "never", "dropped"):
        lat = E.Lattice2D((nx, ny), "f64")
        E.elbm2d_set_tensor_uniform(lat.h, [0.03, 0.005, 0.004])
        if when == "never":
            E.elbm2d_set_table_limit(lat.h, 0)
        before = _free()
        E.elbm2d_set_velocity_field(lat.h, u)
        taken = before - _free()
        assert (taken > tables) == (when != "never")
        E.elbm2d_init_equilibrium(lat.h, phi)
        E.elbm2d_step(lat.h, 5)
        if when == "dropped":
            held = _free()
            E.elbm2d_step(lat.h, 1)
            E.elbm2d_set_table_limit(lat.h, tables - 1)
            assert _free() - held > tables - 4 * MB
            E.elbm2d_step(lat.h, 4)
        else:
            E.elbm2d_step(lat.h, 5)
        out = torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
        E.elbm2d_read_populations(lat.h, out)
        torch.cuda.synchronize()
        states.append(out)
        lat.close()
    assert torch.equal(states[0], states[1]) and torch.equal(states[0], states[2])
