"""The fused forward and backward passes of EnergyFunction (FP32 pair terms) and the FP32 derivative kernels at the sizes
where their loops can go wrong: few monomers, even and odd systems, rows that end a warp, chains of one length or mixed,
partial sets of rows, periodic and open."""
import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs
from helpers import oracle_model, random_conformations

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _system(lens, L, seed=3):
    rng = np.random.Generator(np.random.Philox(seed))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    return inputs.System("t", np.array(lens, np.int32), seq, L, k_tors=-0.5)


SYSTEMS = [([3], 0.0), ([4], 0.0), ([5], 0.0), ([32], 0.0), ([33], 0.0), ([34], 0.0), ([64], 0.0), ([65], 0.0), ([96], 0.0),
           ([3, 3], 12.0), ([4, 5], 12.0), ([3, 30], 16.0), ([9] * 8, 30.0), ([10, 3, 20, 7], 24.0), ([16, 17], 0.0), ([9], 8.0)]


@pytest.mark.parametrize("lens,L", SYSTEMS, ids=["-".join(map(str, s[0])) + ("p" if s[1] else "") for s in SYSTEMS])
def test_gradients_of_every_shape(phast, orc, lens, L):
    """FP32 tolerance of the suite (1e-4 of the largest component, floor 1), for the derivative call and for the training
    step on FP32 and FP64 leaves; the two forms of the energies agree with the oracle and so with one another."""
    s = _system(lens, L)
    x = random_conformations(s, 5, seed=sum(lens), d_min=0.9)
    if len(lens) > 1 and L == 0:   # open-space walks all begin at one point: chains apart
        x[:, lens[0]:] += np.array([6.0, 0.0, 0.0])
    m = oracle_model(orc, s)
    ref = [orc.energy_grad(m, xb) for xb in x]
    Eo, go, po = (np.array([r[k] for r in ref]) for k in range(3))
    gmax = np.maximum(1.0, np.abs(go).max(axis=(1, 2)))
    xt = torch.from_numpy(x).cuda()
    E, gx, gf = phast.phast_energy_grad(s, xt, 32)
    E0, none, _ = phast.phast_energy_grad(s, xt, 32, want_xyz=False, want_ff=False)
    assert none is None
    for e in (E, E0):
        assert np.all(np.abs(e.cpu().numpy() - Eo) <= 1e-4 * np.maximum(1.0, np.abs(Eo)))
    assert np.all(np.abs(gx.cpu().numpy() - go).max(axis=(1, 2)) <= 1e-4 * gmax)
    assert np.all(np.abs(gf.cpu().numpy() - po) <= 1e-4 * np.maximum(1.0, np.abs(po)))
    w = np.array([1.0, -2.0, 0.25, 3.0, 1e-3])
    for dtype in (torch.float32, torch.float64):
        xl = xt.to(dtype).requires_grad_()
        p = torch.tensor(phast.ff_params(s), dtype=dtype, device="cuda", requires_grad=True)
        e = phast.energy(xl, p, s)
        (torch.from_numpy(w).cuda() * e).sum().backward()
        assert e.dtype == torch.float64 and xl.grad.dtype == dtype and p.grad.dtype == dtype
        # coordinates rounded to FP32 move a gradient by up to its own FP32 error again
        tol = (2e-4 if dtype == torch.float32 else 1e-4) * gmax
        assert np.all(np.abs(xl.grad.cpu().double().numpy() - w[:, None, None] * go).max(axis=(1, 2)) <= np.abs(w) * tol)
        scale = (np.abs(w)[:, None] * np.maximum(1.0, np.abs(po))).sum(0)
        assert np.all(np.abs(p.grad.cpu().double().numpy() - (w[:, None] * po).sum(0)) <= 2e-4 * scale)


def test_leaves_that_need_no_gradient_and_expanded_ones(phast):
    s = _system([13], 0.0)
    x = torch.from_numpy(random_conformations(s, 9, seed=1)).cuda().float()
    p = torch.tensor(phast.ff_params(s), dtype=torch.float32)            # parameters on the host
    a = x.clone().requires_grad_()
    phast.energy(a, p, s).sum().backward()                              # the gradient of a sum is an expanded scalar
    b, q = x.transpose(0, 1).contiguous().transpose(0, 1).requires_grad_(), p.clone().requires_grad_()   # strided leaf
    phast.energy(b, q, s).sum().backward()
    c = p.clone().requires_grad_()
    phast.energy(x, c, s).sum().backward()
    assert torch.equal(a.grad, b.grad) and torch.equal(c.grad, q.grad) and c.grad.device.type == "cpu"
    empty = torch.empty(0, 13, 3, device="cuda", requires_grad=True)
    phast.energy(empty, c, s).sum().backward()
    assert empty.grad.shape == (0, 13, 3)
    with pytest.raises(phast.PhastError, match="xyz_bits"):
        st = phast._Structs([s])
        phast._check(phast.lib().phast_energy_forward32(st.sys, st.ff, 1, x.data_ptr(), 16, None, 64, x.data_ptr(), None))


def test_batches_beyond_one_wave(phast):
    """Warps that take several conformations: the batch in one call against the same conformations in small calls."""
    s = _system([9, 9], 14.0)
    x = torch.from_numpy(random_conformations(s, 64, seed=2)).cuda().repeat(700, 1, 1)[:44001].contiguous()
    E, gx, gf = phast.phast_energy_grad(s, x, 32)
    Es, gxs, gfs = phast.phast_energy_grad(s, x[:64].contiguous(), 32)
    idx = torch.arange(x.shape[0], device="cuda") % 64
    assert torch.equal(E, Es[idx]) and torch.equal(gx, gxs[idx]) and torch.equal(gf, gfs[idx])
    xl = x.clone().requires_grad_()
    p = torch.tensor(phast.ff_params(s), dtype=torch.float64, device="cuda", requires_grad=True)
    phast.energy(xl, p, s).sum().backward()
    assert torch.equal(xl.grad, gx)
    assert torch.allclose(p.grad, gf.sum(0), rtol=1e-12, atol=1e-9)
