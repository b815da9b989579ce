"""The FP64 sweep path where its rounds and shortcuts can go wrong: groups of every width on systems
down to one pair a move, and displacements at the edges of the minimum image, against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs
from helpers import oracle_model, oracle_muca, random_conformations

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _mixed(lens, L, k_tors, seed=5):
    rng = np.random.Generator(np.random.Philox(seed))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    chains = [inputs.random_saw(n, 1.0, rng) for n in lens]
    xyz0 = inputs.place_chains(chains, L, 1.0, rng) if L > 0 else np.concatenate(chains)
    p = (0.4, 0.2, 0.2, 0.2) if len(lens) > 1 else (0.7, 0.0, 0.0, 0.3)
    return inputs.System("mixed", np.array(lens, np.int32), seq, L, k_tors=k_tors, e_min=-40.0, bin_width=0.05,
                         n_bins=2400, p=p, recompute_every=3, walkers=5, xyz0=xyz0)


SYSTEMS = {"3": lambda: _mixed([3], 0.0, -0.5), "4": lambda: _mixed([4], 0.0, -0.5), "3+17": lambda: _mixed([3, 17], 9.0, -0.5),
           "33+34": lambda: _mixed([33, 34], 30.0, 0.0), "sphere": lambda: dataclasses.replace(inputs.fene_sphere(5), recompute_every=3)}


@pytest.mark.parametrize("name", list(SYSTEMS))
@pytest.mark.parametrize("tpw", [4, 8, 16, 32])
def test_fp64_sweeps_of_every_group_width(phast, orc, name, tpw):
    """Histograms and coordinates equal the oracle's; with FENE bonds (CUDA's log against libm's) decisions
    may differ at near-ties only, so coordinates are compared only there where all decisions agree."""
    s = SYSTEMS[name]()
    ctx = phast.Context(s, pair_precision=64)
    ctx.set_tile(tpw, 64 // tpw)
    lnW = -0.04 * np.arange(s.n_bins) + 0.8 * np.sin(np.arange(s.n_bins) / 17.0)
    hw = ctx.hist_walker_zeros()
    n_sweeps = 12
    ctx.sweep(n_sweeps, torch.from_numpy(lnW).cuda(), hist_walker=hw)
    st = ctx.get_state("cpu")
    torch.cuda.synchronize()
    hw = hw.cpu().numpy().reshape(s.walkers, s.n_bins)
    xyz = st["xyz"].numpy().reshape(s.walkers, s.n_total, 3)
    m, mu = oracle_model(orc, s), oracle_muca(orc, s)
    agree = 0
    for w, seed in enumerate(s.seeds()):
        wk = orc.new_walker(m, mu, s.xyz0, int(seed))
        h, _, _ = orc.sweep_walker(m, mu, lnW, wk, n_sweeps * s.n_total)
        same = np.array_equal(hw[w].astype(np.uint64), h)
        agree += same
        if same or name != "sphere":
            assert same and np.array_equal(xyz[w], wk.xyz), (name, tpw, w)
            assert abs(float(st["E"][w]) - wk.E) <= 1e-9 * max(1.0, abs(wk.E))
    assert agree >= (4 if name == "sphere" else 5)
    ctx.close()


@pytest.mark.parametrize("count", [0, 1, 2, 3, 7])
def test_fp64_delta_at_the_image_edges(phast, orc, count):
    """Chains displaced so that a component of one pair lies on, or an ulp or 2^-20 of it to either side of, an odd
    multiple of half the box (where the nearest count changes; on it both counts give the same distance)."""
    s = _mixed([3, 17], 9.0, -0.5)
    x = random_conformations(s, 24, seed=count)
    for b in range(24):
        edge = (count + 0.5) * s.box_L
        edge = [edge, np.nextafter(edge, 0), np.nextafter(edge, 1e9), edge * (1 - 2.0 ** -20), edge * (1 + 2.0 ** -20), edge * (1 + 1e-3)][b % 6]
        c = b % 3
        x[b, :3, c] += (x[b, 10, c] - x[b, 1, c]) + (edge if b % 2 else -edge)
    moves = [dict(type=(0, 1, 2, 3)[b % 4], chain=b % 2, index=1, axis=(0.6, 0.0, 0.8), angle=0.3, disp=(0.1, -0.2, 0.3)) for b in range(24)]
    dE = phast.phast_delta_energy(s, torch.from_numpy(x).cuda(), moves).cpu().numpy()
    m = oracle_model(orc, s)
    for b, mv in enumerate(moves):
        o = orc.make_move(mv["type"], mv["chain"], 1, mv["axis"], mv["angle"], mv["disp"])
        ref, _ = orc.delta_energy(m, x[b], o)
        assert abs(dE[b] - ref) <= 1e-10 * max(1.0, orc.delta_scale(m, x[b], o)), (b, dE[b], ref)
