"""The per-node step at the edges of its blocks of 64 nodes: lattices with fewer nodes than a block, one
more and one less than whole blocks, and sides of one and two, against the oracle in every storage."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from gpu_helpers import gpu_lattice, read_pops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec, tol", [("f64", 1e-13), ("f32", 2e-6), ("f16dev", 3e-4), ("bf16dev", 3e-3)])
@pytest.mark.parametrize("dims", [(1, 1, 1), (9, 7, 1), (2, 32, 1), (13, 5, 1), (63, 1, 2), (1, 3, 43), (257, 2, 2)])
@pytest.mark.parametrize("walls", [False, True])
def test_block_edges(dims, prec, tol, walls):
    """One step: the roundings of one collision relative to the largest population (FP16 and BF16
    deviations: 2^-11 and 2^-8 of a deviation of 0.2, twice)."""
    from paper_2605_01774_gb300 import elbm as E
    rng = np.random.default_rng(sum(dims))
    phi0 = 1.0 + 0.2 * rng.uniform(-1, 1, dims[::-1])
    u = (0.0, 0.0, 0.0) if walls else (0.05, -0.03, 0.02)
    D = synth.tensor_from_principal((0.05, 0.01, 0.002), synth.rot_zyz(0.3, 0.7, 1.1))
    bc = (1.2, 0.8) if walls else None
    lat = gpu_lattice(E, dims, prec, D=D, u=u, bc=bc, theta=3e-4)
    E.elbm_init_equilibrium(lat.h, torch.as_tensor(phi0, device="cuda"))
    E.elbm_step(lat.h, 1)
    g = read_pops(E, lat)
    lat.close()
    prob = O.Problem(u=torch.as_tensor(u, dtype=torch.float64), S=O.relaxation_matrix(torch.as_tensor(D)), theta=3e-4,
                     dirichlet_x=bc, lam_mode="reduced")
    ref = O.step(O.init_equilibrium(phi0, torch.as_tensor(u, dtype=torch.float64)), prob, 0)
    assert ((g - ref).abs().max() / ref.abs().max()).item() < tol
