"""Steps launched one after another without waiting (launch.cuh: several may stand on the chip at once,
each reading what the one before wrote) against the same steps with the GPU waited for after each."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
STEPS = 60


@pytest.fixture(scope="module")
def E():
    from paper_2605_01774_gb300 import elbm
    elbm.lib()
    return elbm


def _phi0(dims):
    z, y, x = np.meshgrid(*[np.arange(n) for n in dims[::-1]], indexing="ij")
    return 1 + 0.3 * np.sin(2 * np.pi * x / dims[0]) * np.cos(2 * np.pi * (y / dims[1] + z / dims[2]))


@pytest.mark.parametrize("form", ["still", "moving", "source", "velocity"])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("dims, variant", [((6, 5, 3), 1), ((24, 24, 24), 1), ((32, 20, 12), 2), ((40, 11, 9), 2),
                                           ((32, 20, 12), 3)])
def test_lattice_steps(E, dims, variant, prec, form):
    n = int(np.prod(dims))
    states = []
    for together in (True, False):
        lat = E.Lattice(dims, prec)
        E.elbm_set_tensor_uniform(lat.h, [0.05, 0.01, 0.0, 0.03, 0.005, 0.02])
        if form == "velocity":
            u = 0.03 * np.random.default_rng(1).uniform(-1, 1, (3,) + dims[::-1])
            E.elbm_set_velocity_field(lat.h, torch.as_tensor(u, dtype=torch.float32, device="cuda"))
        else:
            E.elbm_set_velocity_uniform(lat.h, (0.0, 0.0, 0.0) if form == "still" else (0.05, 0.03, 0.02))
        if form == "source":
            E.elbm_set_source(lat.h, (1e-4 * np.random.default_rng(2).random(n)).astype(np.float32))
        try:
            E.elbm_set_step_kernel(lat.h, variant)
        except E.ElbmError as e:
            assert e.status == 9                       # not for this storage and row length
            lat.close()
            pytest.skip("no such step kernel here")
        phi0 = torch.as_tensor(_phi0(dims), device="cuda")
        out = torch.empty((27, n), dtype=torch.float64, device="cuda")
        E.elbm_init_equilibrium(lat.h, phi0)
        if together:
            E.elbm_step(lat.h, STEPS)
        else:
            E.elbm_synchronize(lat.h)
            for _ in range(STEPS):
                E.elbm_step(lat.h, 1)
                E.elbm_synchronize(lat.h)
        E.elbm_read_populations(lat.h, out)
        torch.cuda.synchronize()
        states.append(out.cpu())
        lat.close()
    assert torch.equal(states[0], states[1])


@pytest.mark.parametrize("fields", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", [(7, 5), (90, 40), (128, 64)])
def test_d2q9_steps(E, dims, prec, fields):
    n = dims[0] * dims[1]
    y, x = np.meshgrid(np.arange(dims[1]), np.arange(dims[0]), indexing="ij")
    phi0 = torch.as_tensor(1 + 0.3 * np.sin(2 * np.pi * (x / dims[0] + y / dims[1])), device="cuda")
    states = []
    for together in (True, False):
        lat = E.Lattice2D(dims, prec)
        E.elbm2d_set_tensor_uniform(lat.h, [0.03, 0.005, 0.01])
        if fields:
            u = 0.04 * np.random.default_rng(1).uniform(-1, 1, (2,) + dims[::-1])
            E.elbm2d_set_velocity_field(lat.h, torch.as_tensor(u, dtype=torch.float32, device="cuda"))
        else:
            E.elbm2d_set_velocity_uniform(lat.h, [0.04, 0.01])
        out = torch.empty((9, n), dtype=torch.float64, device="cuda")
        E.elbm2d_init_equilibrium(lat.h, phi0)
        if together:
            E.elbm2d_step(lat.h, STEPS)
        else:
            E.elbm2d_synchronize(lat.h)
            for _ in range(STEPS):
                E.elbm2d_step(lat.h, 1)
                E.elbm2d_synchronize(lat.h)
        E.elbm2d_read_populations(lat.h, out)
        torch.cuda.synchronize()
        states.append(out.cpu())
        lat.close()
    assert torch.equal(states[0], states[1])


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", [(6, 5, 4), (24, 20, 18)])
def test_adjoint_steps(E, dims, prec):
    """The last state of a forward sweep against single steps, each waited for, by the misfit with that
    state's phi as the target: equal to the roundings of the start (1e-13 and 1e-6 of phi; one step
    changes it by 1e-3)."""
    real = torch.float64 if prec == "f64" else torch.float32
    N = int(np.prod(dims))
    theta = torch.zeros((6, N), dtype=real, device="cuda")
    theta[:3] = torch.log(torch.tensor([1e-2, 3e-3, 1e-3], dtype=real, device="cuda"))[:, None]
    theta[3:] = 0.4
    u = [0.02, 0.01, 0.0]
    phi0 = torch.as_tensor(_phi0(dims), device="cuda").to(real).reshape(N)
    h = E.elbm_adjoint_create(dims, prec)
    E.elbm_adjoint_configure(h, u, 1e-8 if prec == "f64" else 3e-4, 7)
    E_i = torch.as_tensor(_equilibrium(u), device="cuda")
    g = (phi0[None] * E_i.to(real)[:, None]).contiguous()
    nxt = torch.empty_like(g)
    for _ in range(STEPS):
        E.elbm_adjoint_step(h, theta, g, None, nxt)
        torch.cuda.synchronize()
        g, nxt = nxt, g
    phi = g.sum(0)
    J, _ = E.elbm_adjoint_misfit(h, theta, phi0, STEPS, [STEPS], phi[None].contiguous(), None)
    E.elbm_adjoint_destroy(h)
    assert (2 * J) ** 0.5 < (1e-13 if prec == "f64" else 1e-6) * float(phi.double().norm())


def _equilibrium(u):
    c = np.array([(a, b, d) for a in (-1, 0, 1) for b in (-1, 0, 1) for d in (-1, 0, 1)], float)
    n = (c != 0).sum(1)
    w = np.array([8 / 27, 2 / 27, 1 / 54, 1 / 216])[n]
    cu, uu = c @ np.array(u), float(np.dot(u, u))
    return w * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
