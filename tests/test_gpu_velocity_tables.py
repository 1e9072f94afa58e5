"""Velocity fields whose nodes lie on both sides of the range in which the equilibrium tables are
summed as a series (extreme c.u near the range's ends), and nodes with phi not above the guard."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu


# |ux| + |uy| + |uz| of equal components: the lower end of the range is at 0.2159
@pytest.mark.parametrize("m", [0.0, 0.1, 0.2150, 0.2158, 0.2160, 0.2200, 0.3, 0.4])
@pytest.mark.parametrize("dims", [(7, 5, 3), (64, 1, 2)])
def test_step_across_the_series_range(m, dims):
    from paper_2605_01774_gb300 import elbm as E
    rng = np.random.default_rng(int(1e4 * m))
    shape = dims[::-1]
    sign = rng.choice([-1.0, 1.0], size=(3,) + shape)
    u = (m / 3 * sign).astype(np.float32)
    u[:, 0, 0, 0] = 0.0
    phi0 = 0.5 + rng.uniform(0, 1, shape)
    ut = torch.as_tensor(u.astype(np.float64))
    g = O.init_equilibrium(phi0, ut) * (1 + 0.05 * torch.as_tensor(rng.standard_normal((27,) + shape)))
    g = g.float().double()
    D = np.diag([0.05, 0.01, 0.002])
    lat = E.Lattice(dims, "f32")
    E.elbm_set_tensor_uniform(lat.h, synth.d6_from_matrix(D))
    E.elbm_set_velocity_field(lat.h, torch.as_tensor(u, device="cuda"))
    E.elbm_set_params(lat.h, theta=3e-4)
    E.elbm_write_populations(lat.h, g.cuda().contiguous())
    E.elbm_step(lat.h, 1)
    out = torch.empty((27,) + shape, dtype=torch.float64, device="cuda")
    E.elbm_read_populations(lat.h, out)
    torch.cuda.synchronize()
    lat.close()
    prob = O.Problem(u=ut, S=O.relaxation_matrix(torch.as_tensor(D)), theta=3e-4, lam_mode="reduced")
    ref = O.step(g, prob, 0)
    # the collision's 30 roundings of 6e-8 of the largest population, and kappa (its sums hold dh, 5 %
    # of g at 20 x 6e-8) times dh
    assert ((out.cpu() - ref).abs().max() / ref.abs().max()).item() < 2e-6
