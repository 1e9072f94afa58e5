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


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_adjoint_states(E, prec):
    """40 steps of 48 x 40 x 44 nodes: 42 states (0.38 or 0.77 GB) by default; with a workspace of 0 only
    checkpoints, in memory that is given back with the call; set afterwards, what is held is given back.
    J and the gradient are bit-equal."""
    dims, steps, every = (48, 40, 44), 40, 8
    real = torch.float64 if prec == "f64" else torch.float32
    shape = dims[::-1]
    state = 27 * dims[0] * dims[1] * dims[2] * (8 if prec == "f64" else 4)
    gen = torch.Generator(device="cuda").manual_seed(4)
    th = torch.empty((6,) + shape, dtype=real, device="cuda").uniform_(-6.0, -3.0, generator=gen)
    phi0 = 1.0 + torch.rand(shape, generator=gen, dtype=real, device="cuda")
    targets = torch.full((1,) + shape, 1.5, dtype=real, device="cuda")
    res = []
    for limit in (None, 0, 20 * state):
        h = E.elbm_adjoint_create(dims, prec)
        E.elbm_adjoint_configure(h, [0.02, 0.0, 0.01], 1e-8 if prec == "f64" else 3e-4, every)
        if limit is not None:
            E.elbm_adjoint_set_workspace(h, limit)
        grad = torch.empty_like(th)
        before = _free()
        J, _ = E.elbm_adjoint_misfit(h, th, phi0, steps, [steps], targets, grad)
        held = before - _free()
        if limit is None:
            assert held >= (steps + 2) * state
            E.elbm_adjoint_set_workspace(h, 0)
            assert before - _free() < 4 * MB
        elif limit == 0:
            assert held < 4 * MB
        else:
            assert held < limit + 4 * MB
        E.elbm_adjoint_destroy(h)
        res.append((J, grad))
    for J, grad in res[1:]:
        assert J == res[0][0] and torch.equal(grad, res[0][1])
