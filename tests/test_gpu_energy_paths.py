"""FP64 energies around the edges of their two paths: system sizes about the smallest that takes far pairs in
double-float, boxes so small that many image counts are not settled in FP32, pairs at the distance where the paths part,
coordinates far from the origin, chains of every mix.  Tolerance: the suite's 1e-11 for FP64 energies."""
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


def _system(lens, L, k_tors=-0.5):
    rng = np.random.Generator(np.random.Philox(17))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    return inputs.System("e", np.array(lens, np.int32), seq, L, k_tors=k_tors)


SYSTEMS = [([3], 0.0), ([4], 0.0), ([30], 0.0), ([33], 0.0), ([47], 0.0), ([48], 0.0), ([49], 0.0), ([3] * 16, 30.0), ([24, 25], 9.0),
           ([24, 24], 8.5), ([20, 41, 3], 0.0), ([100], 0.0), ([32] * 16, 60.0)]


@pytest.mark.parametrize("lens,L", SYSTEMS, ids=["%d-%d%s" % (len(s[0]), sum(s[0]), "p" if s[1] else "") for s in SYSTEMS])
def test_fp64_energies_of_every_size(phast, orc, lens, L):
    s = _system(lens, L)
    if L == 9.0 or L == 8.5:   # too dense for the placing helper: walks laid side by side, many images on the edge
        rng = np.random.default_rng(4)
        x = np.stack([np.concatenate([inputs.random_saw(n, 1.0, rng) + np.array([L / 2 * i, 0.37 * i, 0.2 * i]) for i, n in enumerate(lens)])
                      for _ in range(7)])
    else:
        x = random_conformations(s, 7 if sum(lens) < 300 else 2, seed=sum(lens))
        if L == 0 and len(lens) > 1:
            x[:, lens[0]:] += np.array([5.0, 0.0, 0.0])
            x[:, lens[0] + lens[1]:] += np.array([0.0, 40.0, 0.0])
    x[1] += 1.0e5                                          # far from the origin
    E = phast.phast_energy(s, torch.from_numpy(x).cuda()).cpu().numpy()
    m = oracle_model(orc, s)
    ref = np.array([orc.energy(m, xb) for xb in x])
    assert np.all(np.isfinite(ref))
    assert np.all(np.abs(E - ref) <= 1e-11 * np.maximum(1.0, np.abs(ref))), np.abs(E - ref)


@pytest.mark.parametrize("L", [0.0, 8.0, 25.0])
def test_pairs_where_the_paths_part(phast, orc, L):
    """Two straight chains set so that pairs lie at distance 4, an ulp and 1e-7 to either side, and (L = 8) on the image's
    edge; and coincident monomers, whose energy is infinite."""
    n = 30
    s = _system([n, n], L, k_tors=0.0)
    x = np.stack([np.concatenate([inputs.straight_chain(n, (0, 0, 0), (0, 0, 1)), inputs.straight_chain(n, (r, 0, 0), (0, 0, 1))])
                  for r in (4.0, np.nextafter(4.0, 0), np.nextafter(4.0, 9), 4.0 - 1e-7, 4.0 + 1e-7, 3.0, 11.9, 12.0, 1.0e7 + 3.0)])   # (1e7 itself is a whole number of boxes of 8: coincident)
    E = phast.phast_energy(s, torch.from_numpy(x).cuda()).cpu().numpy()
    m = oracle_model(orc, s)
    ref = np.array([orc.energy(m, xb) for xb in x])
    assert np.all(np.abs(E - ref) <= 1e-11 * np.maximum(1.0, np.abs(ref))), (E, ref)
    x[0, n:] = x[0, :n]
    assert phast.phast_energy(s, torch.from_numpy(x[:1]).cuda()).item() == np.inf


@pytest.mark.parametrize("n", [40, 47, 48, 60, 130])
@pytest.mark.parametrize("bits", [64, 32])
def test_the_wall_stands_whatever_the_other_terms_are(phast, n, bits):
    """A monomer beyond the container's wall: +inf, also where the other terms of the configuration are NaN."""
    rng = np.random.default_rng(2)
    s = inputs.System("w", np.array([n], np.int32), inputs.random_sequence(n, 0.5, np.random.Generator(np.random.Philox(1))), 0.0,
                      k_tors=-0.5, sphere_R=60.0)
    x = np.array([inputs.random_saw(n, 0.9, rng) for _ in range(4)])
    x[0, n // 2] = np.nan
    x[1, 3] += 1000.0
    x[1, n - 3] = np.nan
    x[2, n - 1] += 1000.0
    E = phast.phast_energy(s, torch.from_numpy(x).cuda(), bits).cpu().numpy()
    assert np.all(E[:3] == np.inf) and np.isfinite(E[3])


@pytest.mark.parametrize("lens,L", [([13], 0.0), ([60], 0.0), ([33, 20], 0.0), ([9, 9], 14.0)], ids=["13", "60", "33-20", "9-9p"])
def test_couplings_that_differ_for_ab_and_ba(phast, orc, lens, L):
    """C_LJ with AB unlike BA (the ABI takes four values): FP64 energies and derivatives give a pair the earlier monomer's letter
    first, whatever order the pairs come in; the FP32 derivative kernels give one energy with and without gradients."""
    import dataclasses
    s = dataclasses.replace(_system(lens, L), C=(1.0, -0.5, 0.7, 0.5))
    x = random_conformations(s, 4, seed=sum(lens))
    if L == 0 and len(lens) > 1:
        x[:, lens[0]:] += np.array([6.0, 0.0, 0.0])
    m, xt = oracle_model(orc, s), torch.from_numpy(x).cuda()
    ref = np.array([orc.energy(m, xb) for xb in x])
    tol = 1e-11 * np.maximum(1.0, np.abs(ref))
    assert np.all(np.abs(phast.phast_energy(s, xt).cpu().numpy() - ref) <= tol)
    E, gx, _ = phast.phast_energy_grad(s, xt, 64)
    assert np.all(np.abs(E.cpu().numpy() - ref) <= tol)
    h = 1e-5   # the gradient is that of the energy: central differences of step 1e-5, error under h^2 E''' and 1e-11 E / h
    for j in (0, 5, s.n_total - 1):
        for k in range(3):
            d = np.zeros_like(x)
            d[:, j, k] = h
            num = np.array([orc.energy(m, a) - orc.energy(m, b) for a, b in zip(x + d, x - d)]) / (2 * h)
            assert np.all(np.abs(gx[:, j, k].cpu().numpy() - num) <= 1e-4 * np.maximum(1.0, np.abs(num)))
    E1 = phast.phast_energy_grad(s, xt, 32)[0].cpu().numpy()
    E0 = phast.phast_energy_grad(s, xt, 32, want_xyz=False, want_ff=False)[0].cpu().numpy()
    assert np.all(np.abs(E1 - E0) <= 1e-4 * np.maximum(1.0, np.abs(E1)))
    c = (-0.5 + 0.7) / 2 if len(lens) == 1 else -0.5   # the one value that the FP32 kernels take for AB and BA
    m32 = oracle_model(orc, dataclasses.replace(s, C=(1.0, c, c, 0.5)))
    r32 = np.array([orc.energy(m32, xb) for xb in x])
    assert np.all(np.abs(E1 - r32) <= 1e-4 * np.maximum(1.0, np.abs(r32)))


EXTENDED = [("walks", [60], 0.0, {}, 0.0, 1.0, 0.0), ("longer walks", [150], 0.0, {}, 0.0, 1.0, 0.0),
            ("blown up", [60], 0.0, dict(k_bend=0.0), 0.0, 8.0, 0.0), ("blown up far", [60], 0.0, dict(k_bend=0.0), 0.0, 1.0e4, 0.0),
            ("chains from afar", [60, 60], 0.0, dict(k_bend=0.0, k_lj_intra=0.0), 60.0, 1.0, 0.0),
            ("chains from afar in a box", [60, 60], 300.0, dict(k_bend=0.0, k_lj_intra=0.0), 60.0, 1.0, 0.0),
            ("1e9 out", [60], 0.0, {}, 0.0, 1.0, 1.0e9), ("1e12 out", [60], 0.0, {}, 0.0, 1.0, 1.0e12),
            ("chains 1e12 out", [30, 30], 0.0, {}, 6.0, 1.0, 1.0e12)]


def _extended(s, x):
    """Energy of configurations x in extended precision: bending and Lennard-Jones terms, and the sum of their sizes."""
    x = x.astype(np.longdouble)
    off = np.concatenate([[0], np.cumsum(s.chain_len)])
    chain = np.repeat(np.arange(len(s.chain_len)), s.chain_len)
    terms = []
    for c in range(len(s.chain_len)):
        b = np.diff(x[:, off[c]:off[c + 1]], axis=1)
        l = np.sqrt((b * b).sum(2))
        terms.append(np.longdouble(s.k_bend) * (1 - (b[:, 1:] * b[:, :-1]).sum(2) / (l[:, 1:] * l[:, :-1])))
    i, j = np.triu_indices(s.n_total, 1)
    keep = ~((chain[i] == chain[j]) & (j == i + 1))
    i, j = i[keep], j[keep]
    d, inter = x[:, i] - x[:, j], chain[i] != chain[j]
    if s.box_L > 0:
        L = np.longdouble(s.box_L)
        d = np.where(inter[None, :, None], d - L * np.rint(d / L), d)
    i6 = 1 / (d * d).sum(2) ** 3
    k = np.where(inter, np.longdouble(s.k_lj_inter), np.longdouble(s.k_lj_intra))
    terms.append(k * (i6 * (i6 - np.array(s.C, np.longdouble)[2 * s.seq[i].astype(int) + s.seq[j]])))
    t = np.concatenate(terms, axis=1)
    return t.sum(1), np.abs(t).sum(1)


@pytest.mark.parametrize("name,lens,L,kw,gap,scale,out", EXTENDED, ids=[e[0].replace(" ", "-") for e in EXTENDED])
def test_fp64_energies_to_the_last_digits(phast, name, lens, L, kw, gap, scale, out):
    """Against extended precision: within 16 FP64 roundings of the sum of the terms' sizes (a term has about a dozen, a lane's
    sum of n / 128 terms and the tree a few more, all of them independent), also where far pairs are all there is and for
    conformations far from the origin."""
    s = _system(lens, L, k_tors=0.0)
    for k, v in kw.items():
        setattr(s, k, v)
    rng = np.random.default_rng(1)
    x = np.array([np.concatenate([inputs.random_saw(n, 0.9, rng) + np.array([gap * i, 0.0, 0.0]) for i, n in enumerate(lens)])
                  for _ in range(12)]) * scale + out
    E = phast.phast_energy(s, torch.from_numpy(x).cuda()).cpu().numpy().astype(np.longdouble)
    ref, size = _extended(s, x)
    assert np.all(np.abs(E - ref) <= 16 * 2.0 ** -53 * size), ((E - ref) / size / 2.0 ** -53).astype(float)


@pytest.mark.parametrize("lens,L", [([5], 0.0), ([33, 20], 0.0), ([9, 9], 14.0)], ids=["5", "33-20", "9-9p"])
@pytest.mark.parametrize("bits", [64, 32])
def test_energy_changes_of_configurations_that_have_no_energy(phast, lens, L, bits):
    """A coordinate that is infinite or NaN: the change of a move elsewhere is NaN."""
    s = _system(lens, L)
    x = random_conformations(s, 4, seed=3)
    if L == 0 and len(lens) > 1:
        x[:, lens[0]:] += np.array([6.0, 0.0, 0.0])
    x[1, 0, 1], x[2, 0, 0], x[3, 0, 2] = np.inf, -np.inf, np.nan
    c = len(lens) - 1
    move = dict(type=0, chain=c, index=lens[c] - 2, axis=np.array([0.0, 0.6, 0.8]), angle=0.05)
    dE = phast.phast_delta_energy(s, torch.from_numpy(x).cuda(), [move] * 4, bits).cpu().numpy()
    assert np.isfinite(dE[0]) and np.all(np.isnan(dE[1:])), dE
    if len(lens) == 1:   # a rotation of the only chain changes no pair
        whole = dict(type=2, chain=0, index=0, axis=np.array([0.0, 0.6, 0.8]), angle=0.05)
        assert np.all(phast.phast_delta_energy(s, torch.from_numpy(x).cuda(), [whole] * 4, bits).cpu().numpy()[:3] == 0.0)


@pytest.mark.parametrize("bond,L", [(1.0e5, 12.0), (1.0e3, 37.0), (30.0, 12.0)])
def test_unwrapped_chains_many_boxes_long(phast, bond, L):
    """Displacements of up to 1e6 between chains come down to half a box by their images: to the rounding of the FP64 coordinates'
    differences (2 x 2^-53 of the largest in each component, 12 / r of a pair) and 16 roundings of the terms."""
    s = _system([24, 25, 20], L, k_tors=0.0)
    rng = np.random.default_rng(1)
    x = np.array([np.concatenate([inputs.random_saw(n, 0.9, rng) + np.array([0.3, 0.2, 0.4]) * i for i, n in enumerate(s.chain_len)])
                  for _ in range(12)]) * bond
    E = phast.phast_energy(s, torch.from_numpy(x).cuda()).cpu().numpy().astype(np.longdouble)
    ref, size = _extended(s, x)
    chain = np.repeat(np.arange(3), s.chain_len)
    i, j = np.triu_indices(s.n_total, 1)
    i, j = i[chain[i] != chain[j]], j[chain[i] != chain[j]]
    d = x[:, i] - x[:, j]
    r = np.sqrt(((d - L * np.rint(d / L)) ** 2).sum(2))
    steep = (s.k_lj_inter * (12 * r ** -12.0 + 6 * r ** -6.0) / r).sum(1)   # |dE / dr| of the pairs between chains
    assert np.all(np.abs(E - ref) <= 16 * 2.0 ** -53 * size + 2 * 3 ** 0.5 * 2.0 ** -53 * np.abs(x).max(axis=(1, 2)) * steep)


@pytest.mark.parametrize("n", [48, 55, 200, 512])
@pytest.mark.parametrize("direction", [(1.0, 0.0, 0.0), (1.0, 1.0, 1.0), (0.3, -0.5, 0.9)], ids=["axis", "diagonal", "oblique"])
def test_straight_chains_to_the_last_digits(phast, n, direction):
    """No bending and the fewest near pairs that an ordinary chain can have, so that far pairs weigh most: the bound of
    test_fp64_energies_to_the_last_digits, for stretched and slightly bent chains."""
    s = _system([n], 0.0, k_tors=0.0)
    rng = np.random.default_rng(n)
    x = np.array([inputs.straight_chain(n, direction=direction) * r + rng.normal(size=(n, 3)) * e for r in (1.0, 1.3) for e in (0.0, 1e-3, 0.05)])
    E = phast.phast_energy(s, torch.from_numpy(x).cuda()).cpu().numpy().astype(np.longdouble)
    ref, size = _extended(s, x)
    assert np.all(np.abs(E - ref) <= 16 * 2.0 ** -53 * size), ((E - ref) / size / 2.0 ** -53).astype(float)
