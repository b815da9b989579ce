"""FP32 derivative kernels on conformations spread far out: left-out pairs and the stand-ins of rows and partners that do not
exist must add nothing, wherever the monomers are and however small the real terms.  Tolerance: the suite's 1e-4 of FP32 pair
terms, here of the value itself; where the centroid of a chain is a distance c from its near monomers, FP32 coordinates about it
are rounded by c 2^-24 each, which moves a contact's force by 14/r of the pair's error."""
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


def _system(lens, L=0.0, **kw):
    rng = np.random.Generator(np.random.Philox(17))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    return inputs.System("f", np.array(lens, np.int32), seq, L, **kw)


def _check(phast, orc, s, x, c=0.0):
    tol = max(1e-4, 14 / 0.9 * 2 * 3 ** 0.5 * c * 2.0 ** -24)
    m, xt = oracle_model(orc, s), torch.from_numpy(x).cuda()
    ref = [orc.energy_grad(m, xb) for xb in x]
    Eo, go = (np.array([r[k] for r in ref]) for k in range(2))
    E, gx, _ = phast.phast_energy_grad(s, xt, 32)
    E0 = phast.phast_energy_grad(s, xt, 32, want_xyz=False, want_ff=False)[0]
    for e in (E, E0):
        assert np.all(np.abs(e.cpu().numpy() - Eo) <= 1e-4 * np.abs(Eo)), (e, Eo)
    assert np.all(np.abs(gx.cpu().numpy() - go).max(axis=(1, 2)) <= tol * np.abs(go).max(axis=(1, 2)))


@pytest.mark.parametrize("lens", [[9], [13], [32], [33], [65], [9, 9], [13, 8, 3]], ids=lambda v: "-".join(map(str, v)))
@pytest.mark.parametrize("far", [1.0e4, -1.0e4])
def test_a_monomer_far_from_its_chain(phast, orc, lens, far):
    """The first monomer 1e4 from the chain's origin in each component (the middle monomer's FP32 value, or the centroid)."""
    s = _system(lens)
    rng = np.random.default_rng(1)
    x = np.concatenate([inputs.random_saw(n, 0.9, rng) + np.array([6.0 * i, 0.0, 0.0]) for i, n in enumerate(lens)])[None]
    n = lens[0]
    x[0, 0] = x[0, n // 2].astype(np.float32) + far if len(lens) == 1 else x[0, 1:n].mean(0) + far * n / (n - 1)
    _check(phast, orc, s, x, 3 ** 0.5 * abs(far) / (n - 1) if len(lens) > 1 else 0.0)


@pytest.mark.parametrize("scale", [1.0e2, 1.0e3, 1.0e4])
@pytest.mark.parametrize("lens,L", [([20], 0.0), ([33], 0.0), ([11, 9], 0.0), ([11, 9], 3.0e5)], ids=["20", "33", "11-9", "11-9p"])
def test_conformations_blown_up(phast, orc, lens, L, scale):
    """Lennard-Jones terms alone, every distance 1e2 to 1e4 times its usual one (the smallest energies about 1e-24)."""
    s = _system(lens, L, k_bend=0.0)
    rng = np.random.default_rng(1)
    x = np.array([inputs.random_saw(sum(lens), 0.9, rng) for _ in range(4)]) * scale
    _check(phast, orc, s, x)


@pytest.mark.parametrize("bond", [1.0e5, 1.0e7])
@pytest.mark.parametrize("lens,L", [([20], 0.0), ([20], 3.0e9), ([11, 9], 0.0), ([9] * 4, 3.0e9)], ids=["20", "20p", "11-9", "9x4p"])
def test_local_terms_of_long_bonds(phast, orc, lens, L, bond):
    """Bending and torsion alone: the products of squares that their FP32 form takes the root of leave FP32 (the eighth power of a
    bond for the torsion), the terms and gradients do not."""
    s = _system(lens, L, k_tors=-0.5, k_lj_intra=0.0, k_lj_inter=0.0)
    rng = np.random.default_rng(1)
    x = np.array([np.concatenate([inputs.random_saw(n, 0.9, rng) + np.array([12.0 * i, 0.0, 0.0]) for i, n in enumerate(lens)])
                  for _ in range(4)]) * bond
    _check(phast, orc, s, x)
