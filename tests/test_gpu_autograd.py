"""phast.energy's backward pass where its incoming gradient is more than a tensor of values: differentiated again (jvp by two
backward passes, create_graph), batched (vectorised Jacobians), with a forward-mode tangent; and saved tensors that come back in
another type.  dE/dx of phast_energy_grad is the reference: the same kernels, so FP64 leaves agree to the rounding of a sum and
FP32 ones to that of FP32."""
import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs
from helpers import random_conformations

pytestmark = pytest.mark.gpu
RTOL = {torch.float64: 1e-12, torch.float32: 1e-5}


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


@pytest.fixture(scope="module", params=[(torch.float64, 32), (torch.float32, 32), (torch.float64, 64)], ids=["x64", "x32", "pairs64"])
def case(request, phast):
    dtype, pairs = request.param
    s = inputs.System("a", np.array([13], np.int32), inputs.fibonacci_sequence(13), 0.0, k_tors=-0.5)
    x = torch.from_numpy(random_conformations(s, 4, seed=5)).cuda().to(dtype)
    p = torch.tensor(phast.ff_params(s), dtype=dtype, device="cuda")
    _, gx, gf = phast.phast_energy_grad(s, x.double(), pairs)
    return s, x, p, gx, gf, pairs


def _close(a, b, dtype):
    assert a.shape == b.shape and torch.all((a.double() - b).abs() <= RTOL[dtype] * b.abs().max())


def test_jvp_by_two_backward_passes(phast, case):
    s, x, p, gx, gf, pairs = case
    v = torch.randn(x.shape, dtype=x.dtype, generator=torch.Generator().manual_seed(1)).cuda()
    u = torch.randn(5, dtype=x.dtype, generator=torch.Generator().manual_seed(2)).cuda()
    _, jv = torch.autograd.functional.jvp(lambda y, q: phast.energy(y, q, s, pairs), (x, p), (v, u), strict=True)
    _close(jv, (gx * v.double()).sum((1, 2)) + gf @ u.double(), x.dtype)


def test_vectorised_jacobian(phast, case):
    s, x, p, gx, gf, pairs = case
    J, Jp = torch.autograd.functional.jacobian(lambda y, q: phast.energy(y, q, s, pairs), (x, p), vectorize=True)
    B = x.shape[0]
    full = torch.zeros(B, *x.shape, dtype=torch.float64, device="cuda")
    full[torch.arange(B), torch.arange(B)] = gx
    _close(J, full, x.dtype)
    _close(Jp, gf, x.dtype)


def test_gradient_of_a_function_of_the_energies_keeps_its_graph(phast, case):
    """d/dE of (E^2)' is 2 in the expression that the gradient is linear in."""
    s, x, p, gx, gf, pairs = case
    y = x.clone().requires_grad_()
    e = phast.energy(y, p, s, pairs)
    w = torch.ones_like(e, requires_grad=True)
    g, = torch.autograd.grad(e, y, grad_outputs=w, create_graph=True)
    assert g.requires_grad
    d, = torch.autograd.grad((g.double() * gx).sum(), w)
    _close(d, (gx * gx).sum((1, 2)), x.dtype)


def test_forward_mode_tangent_of_the_incoming_gradient(phast, case):
    s, x, p, gx, gf, pairs = case
    y = x.clone().requires_grad_()
    e = phast.energy(y, p, s, pairs)
    t = torch.tensor([1.0, -2.0, 0.5, 3.0], dtype=torch.float64, device="cuda")
    with torch.autograd.forward_ad.dual_level():
        g, = torch.autograd.grad(e, y, grad_outputs=torch.autograd.forward_ad.make_dual(torch.ones_like(t), t))
        tangent = torch.autograd.forward_ad.unpack_dual(g).tangent
        assert tangent is not None
        _close(tangent, t.view(-1, 1, 1) * gx, x.dtype)


def test_saved_tensors_that_come_back_in_another_type(phast, case):
    """bfloat16 leaves unpacked as FP32 by a hook: the conformations that bfloat16 holds."""
    s, x, p, _, _, pairs = case
    y = x.to(torch.bfloat16).requires_grad_()
    gx = phast.phast_energy_grad(s, y.detach().double(), pairs)[1]
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.detach(), lambda t: t.float()):
        e = phast.energy(y, p, s, pairs)
    e.sum().backward()
    assert y.grad.dtype == torch.bfloat16
    assert torch.all((y.grad.double() - gx).abs() <= 2.0 ** -8 * gx.abs() + 1e-5 * gx.abs().max())
