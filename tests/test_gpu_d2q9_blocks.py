"""D2Q9 step: rows in blocks of their own and nodes dealt out in a row give the same bits.  A state that
repeats along x is stepped once as one period (short rows) and once as several (long rows)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nx, copies, ny", [(33, 3, 5), (8, 16, 3), (5, 25, 1), (65, 2, 4), (1, 96, 70), (43, 6, 129)])
@pytest.mark.parametrize("fields", [False, True])
def test_short_and_long_rows_agree(prec, nx, copies, ny, fields):
    from paper_2605_01774_gb300 import elbm as E
    gen = torch.Generator(device="cuda").manual_seed(nx * ny)
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda")  # noqa: E731
    phi, a, b, th = 0.2 + rand(ny, nx), 0.01 + 0.04 * rand(ny, nx), 1e-3 + 1e-3 * rand(ny, nx), 6 * rand(ny, nx)
    c, s = torch.cos(th), torch.sin(th)
    D = torch.stack([c * c * a + s * s * b, c * s * (a - b), s * s * a + c * c * b])
    u = 0.2 * rand(2, ny, nx) - 0.1
    u[:, 0, 0] = 0.0
    out = []
    for k in (1, copies):
        lat = E.Lattice2D((nx * k, ny), prec)
        if fields:
            E.elbm2d_set_tensor_field(lat.h, D.repeat(1, 1, k).contiguous())
            E.elbm2d_set_velocity_field(lat.h, u.repeat(1, 1, k).contiguous())
        else:
            E.elbm2d_set_tensor_uniform(lat.h, [0.03, 0.005, 0.004])
            E.elbm2d_set_velocity_uniform(lat.h, [0.04, 0.01])
        E.elbm2d_init_equilibrium(lat.h, phi.repeat(1, k).contiguous())
        E.elbm2d_step(lat.h, 5)
        g = torch.empty((9, ny, nx * k), dtype=torch.float64, device="cuda")
        E.elbm2d_read_populations(lat.h, g)
        torch.cuda.synchronize()
        out.append(g)
        lat.close()
    assert torch.equal(out[0].repeat(1, 1, copies), out[1])


@pytest.mark.parametrize("at_rest", [False, True])
def test_tables_kept_or_formed_in_the_step(at_rest):
    """FP64 velocity fields: 50 x 55 nodes keep their tables; as 110 x 100 repeats (8.7 GB of tables, above
    the limit) they are formed in every step.  The bits are the same."""
    from paper_2605_01774_gb300 import elbm as E
    gen = torch.Generator(device="cuda").manual_seed(9)
    phi = 0.2 + torch.rand((55, 50), generator=gen, device="cuda")
    u = 0.3 * torch.rand((2, 55, 50), generator=gen, device="cuda") - 0.15
    u[:, ::3] = 0.0
    if at_rest:
        u.zero_()
    out = []
    for ky, kx in ((1, 1), (100, 110)):
        lat = E.Lattice2D((50 * kx, 55 * ky), "f64")
        E.elbm2d_set_tensor_uniform(lat.h, [0.03, 0.005, 0.004])
        E.elbm2d_set_velocity_field(lat.h, u.repeat(1, ky, kx).contiguous())
        E.elbm2d_init_equilibrium(lat.h, phi.repeat(ky, kx).contiguous())
        E.elbm2d_step(lat.h, 3)
        g = torch.empty((9, 55 * ky, 50 * kx), dtype=torch.float64, device="cuda")
        E.elbm2d_read_populations(lat.h, g)
        torch.cuda.synchronize()
        out.append(g)
        lat.close()
    assert torch.equal(out[0], out[1][:, :55, :50]) and torch.equal(out[0], out[1][:, -55:, -50:])
