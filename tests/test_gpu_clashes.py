"""Clashing conformations with FP32 pairs: energies and gradients beyond FP32's range are infinite or the FP64 sum, as they are
with FP64 pairs, and never NaN where the sum has a value."""
import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs
from helpers import oracle_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _system(lens, **kw):
    rng = np.random.Generator(np.random.Philox(17))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    return inputs.System("c", np.array(lens, np.int32), seq, 0.0, k_tors=-0.5, **kw)


def _walks(lens, B):
    rng = np.random.default_rng(1)
    return np.array([np.concatenate([inputs.random_saw(n, 0.9, rng) + np.array([6.0 * i, 0.0, 0.0]) for i, n in enumerate(lens)])
                     for _ in range(B)])


@pytest.mark.parametrize("lens", [[13], [30, 30], [9] * 4], ids=lambda v: "-".join(map(str, v)))
def test_energies_of_clashing_monomers(phast, orc, lens):
    """Coincident monomers, a pair whose energy leaves FP32 (r = 1e-5), and two pairs of 2.5e38 each (r = 7.08e-4), whose
    sum does: +inf, and the sum.  FP32 coordinates of magnitude 4 move r by up to 1.2e-3 of it, the energy by 1.4 %."""
    s = _system(lens)
    x = _walks(lens, 4)
    x[1, -1] = x[1, 2]
    x[2, -1] = x[2, 2] + 1e-5
    x[3, -1] = x[3, 3] + np.array([7.08e-4, 0.0, 0.0])
    x[3, -2] = x[3, 2] + np.array([0.0, 7.08e-4, 0.0])
    xt = torch.from_numpy(x).cuda()
    m = oracle_model(orc, s)
    ref = [orc.energy(m, x[b]) for b in (0, 3)]
    assert 4.0e38 < ref[1] < 6.0e38
    E = phast.phast_energy(s, xt, 32).cpu().numpy()
    assert abs(E[0] - ref[0]) <= 1e-4 * max(1.0, abs(ref[0])) and E[1] == np.inf and E[2] == np.inf
    assert abs(E[3] - ref[1]) <= 0.05 * ref[1]
    for want in (True, False):
        E = phast.phast_energy_grad(s, xt, 32, want_xyz=want, want_ff=want)[0].cpu().numpy()
        assert abs(E[0] - ref[0]) <= 1e-4 * max(1.0, abs(ref[0])) and np.all(E[1:3] == np.inf)
    p = torch.tensor(phast.ff_params(s), dtype=torch.float32, device="cuda")
    assert torch.all(phast.energy(xt.float(), p, s)[1:3] == np.inf)


@pytest.mark.parametrize("lens", [[13], [9, 9]], ids=lambda v: "-".join(map(str, v)))
def test_fp32_gradients_scaled_beyond_the_range(phast, lens):
    """FP32 leaves whose gradient times dloss/dE overflows, is infinite, underflows or comes of a dloss/dE that FP32 does not
    hold: the FP64 product rounded to FP32 (1e-5 of the largest, and the spacing of FP32's subnormals)."""
    s = _system(lens)
    w = torch.tensor([1.0, 1.0, 1e30, 1e41, 1e-42, -3e38, 0.0, 1e-39, -1e-60], dtype=torch.float64, device="cuda")
    x = _walks(lens, len(w))
    x[1, -1] = x[1, 2] + np.array([1e-5, 0.0, 0.0])
    x[2, -1] = x[2, 2] + np.array([3e-3, 0.0, 0.0])
    x[8, -1] = x[8, 2] + np.array([3e-3, 0.0, 0.0])
    y = torch.from_numpy(x).cuda().float().requires_grad_()
    p = torch.tensor(phast.ff_params(s), dtype=torch.float32, device="cuda")
    phast.energy(y, p, s).backward(w)
    gx = phast.phast_energy_grad(s, y.detach().double(), 32)[1]
    ref = (w.view(-1, 1, 1) * gx).float()
    got = y.grad
    assert torch.equal(got.isinf(), ref.isinf()) and torch.equal(got.isnan(), ref.isnan())
    assert ref[1:4].isinf().any(dim=2).any(dim=1).all() and ref[5].isinf().any() and not ref[[0, 2, 3, 4, 5, 6, 7, 8]].isnan().any()
    assert torch.equal(got[got.isinf()], ref[ref.isinf()])
    fin = ref.isfinite()
    for b in range(len(w)):
        g, r = got[b][fin[b]].double(), ref[b][fin[b]].double()
        if r.numel():
            assert torch.all((g - r).abs() <= 1e-5 * r.abs().max() + 2.0 ** -148), b
