"""Paths of the adjoint's kernels at the sizes and values where they change: partial blocks, nodes
that the FP64 fixed-point step hands to FP64 arithmetic, and runs whose states are kept or
recomputed from checkpoints."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
U = np.array([0.02, -0.03, 0.01])


@pytest.fixture(scope="module")
def E():
    from paper_2605_01774_gb300 import elbm
    elbm.lib()
    return elbm


def _state(dims, seed):
    rng = np.random.default_rng(seed)
    shape = tuple(dims[::-1])
    th = np.stack([np.log(d) + 0.3 * rng.standard_normal(shape) for d in (1e-2, 1e-3, 1e-4)]
                  + [rng.uniform(0, 2 * np.pi, shape) for _ in range(3)])
    g = O.init_equilibrium(0.5 + rng.uniform(0, 1, shape), torch.as_tensor(U))
    g = g * (1 + 0.05 * torch.as_tensor(rng.standard_normal(g.shape)))
    return torch.as_tensor(th), g


# a scale of 1e-280 is outside the fixed-point range: every node takes FP64 arithmetic; "mixed": some
# nodes are negligible beside their largest population, some are zero
@pytest.mark.parametrize("dims", [(5, 3, 7), (64, 1, 1), (13, 11, 3)])
@pytest.mark.parametrize("kind", ["plain", "small", "mixed"])
def test_forward_f64(E, dims, kind):
    th, g = _state(dims, 1)
    scale = 1e-280 if kind == "small" else 1.0
    if kind == "mixed":
        flat = g.reshape(27, -1)
        flat[:, ::5] = 0.0
        flat[0, 1::5] = -flat[1:, 1::5].sum(0) * (1 - 1e-6)
    h = E.elbm_adjoint_create(dims, "f64")
    E.elbm_adjoint_configure(h, U, 1e-8, 4)
    out = torch.empty_like(g, device=DEV)
    E.elbm_adjoint_step(h, th.to(DEV), (scale * g).to(DEV).contiguous(), g_next=out)
    E.elbm_adjoint_destroy(h)
    # the collision is homogeneous of degree one; the oracle forms dh^2, which has no value at 1e-560
    S = O.relaxation_matrix(O.tensor_from_params(th))
    ref = O.step(g, O.Problem(u=torch.as_tensor(U), S=S, theta=1e-8), 0)
    # some 60 roundings of 1.1e-16, and the quotient kappa of sums that cancel by 20 (dh is 5 % of g);
    # "mixed" nodes with phi 1e-6 of the largest population lose another factor in kappa
    tol = 2e-13 if kind != "mixed" else 1e-9
    assert ((out.cpu() / scale - ref).abs().max() / ref.abs().max()).item() < tol


@pytest.mark.parametrize("dims", [(5, 3, 7), (128, 1, 1), (43, 3, 1)])
def test_vjp_f32_against_f64(E, dims):
    """FP32 rounds dh = 5 % of g at 20 x 6e-8; some ten such roundings add up: 1e-5, with margin 1e-4."""
    th, g = _state(dims, 2)
    y = torch.as_tensor(np.random.default_rng(3).standard_normal(g.shape))
    res = []
    for prec, t in (("f64", torch.float64), ("f32", torch.float32)):
        h = E.elbm_adjoint_create(dims, prec)
        E.elbm_adjoint_configure(h, U, 3e-4, 4)
        gbar, grad = torch.empty(g.shape, dtype=t, device=DEV), torch.empty(th.shape, dtype=t, device=DEV)
        E.elbm_adjoint_step(h, th.to(DEV, t), g.to(DEV, t).contiguous(), gbar_next=y.to(DEV, t), gbar=gbar, grad6=grad)
        E.elbm_adjoint_destroy(h)
        res.append((gbar.double().cpu(), grad.double().cpu()))
    for a, b in zip(*res):
        assert (torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(a)).item() < 1e-4


@pytest.mark.parametrize("steps, every", [(17, 1), (18, 4), (20, 4), (16, 5)])
def test_states_kept_or_recomputed(E, steps, every):
    """104 x 104 x 100 in FP64 is 234 MB a state: runs of 17 steps and more are checkpointed, those of
    16 and fewer kept (4 GiB).  The states are the same either way, so J and the gradient are
    bit-equal to those of one segment (every = steps)."""
    dims = (104, 104, 100)
    gen = torch.Generator(device=DEV).manual_seed(4)
    shape = dims[::-1]
    th = torch.empty((6,) + shape, dtype=torch.float64, device=DEV).uniform_(-6.0, -3.0, generator=gen)
    phi0 = 1.0 + torch.rand(shape, generator=gen, dtype=torch.float64, device=DEV)
    obs = [steps // 2, steps]
    targets = torch.full((2,) + shape, 1.5, dtype=torch.float64, device=DEV)
    res = []
    for k in (every, steps):
        h = E.elbm_adjoint_create(dims, "f64")
        E.elbm_adjoint_configure(h, U, 1e-8, k)
        grad = torch.empty_like(th)
        J, _ = E.elbm_adjoint_misfit(h, th, phi0, steps, obs, targets, grad6=grad)
        J0, _ = E.elbm_adjoint_misfit(h, th, phi0, steps, obs, targets)
        assert J0 == J
        E.elbm_adjoint_destroy(h)
        res.append((J, grad))
    assert res[0][0] == res[1][0] and torch.equal(res[0][1], res[1][1])
