"""The exact FP64 replay of accepted moves in FP32 sweeps, for groups of every width: chains of 3 to 55 monomers (the
thresholds of the centroid's summation tree and of the few-monomer rotation), random and straight starts (the builds
without and with the exact torsion path), and the recompute period counted across calls."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs
from helpers import oracle_model, oracle_muca

pytestmark = pytest.mark.gpu

LENS = [3, 8, 9, 16, 17, 33, 55]


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _system(straight):
    rng = np.random.Generator(np.random.Philox(12))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in LENS])
    chains = [inputs.straight_chain(n) if straight else inputs.random_saw(n, 1.0, rng) for n in LENS]
    xyz0 = np.concatenate([c + np.array([0.0, 6.0 * i, 0.0]) for i, c in enumerate(chains)]) if straight else \
        inputs.place_chains(chains, 60.0, 1.0, rng)
    return inputs.System("chains", np.array(LENS, np.int32), seq, 60.0, k_tors=-0.5, e_min=-400.0, bin_width=0.5, n_bins=1600,
                         p=(0.3, 0.2, 0.3, 0.2), recompute_every=2, walkers=3, xyz0=xyz0)


@pytest.mark.parametrize("straight", [False, True])
@pytest.mark.parametrize("tpw", [4, 8, 16, 32])
def test_replayed_coordinates_are_the_oracles(phast, orc, tpw, straight):
    """The oracle replays every walker with the GPU's decisions imposed: the coordinates agree bit for bit, and the FP64
    energy that the last move's recompute left in place agrees to rounding."""
    s = _system(straight)
    ctx = phast.Context(s, pair_precision=32)
    ctx.set_tile(tpw, max(1, 32 // tpw))
    n_sweeps, W = 4, s.walkers
    trace = ctx.trace_buffer(n_sweeps, W)
    ctx.sweep(n_sweeps, ctx.lnW_zeros(), trace=trace, trace_walkers=W)
    st = ctx.get_state("cpu")
    torch.cuda.synchronize()
    tr = trace.cpu().numpy().view(phast.TRACE_DTYPE).reshape(W, -1)
    xyz = st["xyz"].numpy().reshape(W, s.n_total, 3)
    m, mu = oracle_model(orc, s), oracle_muca(orc, s)
    for w, seed in enumerate(s.seeds()):
        wk = orc.new_walker(m, mu, s.xyz0, int(seed))
        orc.sweep_walker(m, mu, np.zeros(s.n_bins), wk, n_sweeps * s.n_total, force=tr[w]["accepted"].astype(np.uint8))
        assert np.array_equal(xyz[w], wk.xyz), (tpw, straight, w)
        ref = orc.energy(m, wk.xyz)
        assert abs(float(st["E"][w]) - ref) <= 1e-11 * max(1.0, abs(ref))
    assert np.all(ctx.stats()["recomputes"] == 2)
    ctx.close()


@pytest.mark.parametrize("tile", [(32, 1), (16, 2), (1, 32)])
@pytest.mark.parametrize("precision", [32, 64])
def test_recompute_period_counts_across_calls(phast, tile, precision):
    s = dataclasses.replace(inputs.config1(5), recompute_every=3)
    a, b = (phast.Context(s, pair_precision=precision) for _ in range(2))
    for c, calls in ((a, [10]), (b, [1, 1, 2, 4, 2])):
        c.set_tile(*tile)
        for n in calls:
            c.sweep(n, c.lnW_zeros())
    sa, sb = a.get_state("cpu"), b.get_state("cpu")
    torch.cuda.synchronize()
    assert np.all(a.stats()["recomputes"] == 3) and np.all(b.stats()["recomputes"] == 3)
    if precision == 64:   # FP64 decisions do not depend on where a call ends
        assert torch.equal(sa["xyz"], sb["xyz"]) and torch.equal(sa["bin"], sb["bin"])
    a.close()
    b.close()
