"""One-walker-per-thread tiles: a walker's trajectory does not depend on the tile that it runs in (partly filled warps, trial
records in shared or in global memory, several tiles per SM), and it is the oracle's for the accepted moves."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs
from helpers import oracle_model, oracle_muca

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _system(kind, walkers):
    if kind == "sphere":
        return dataclasses.replace(inputs.fene_sphere(walkers), recompute_every=3)
    rng = np.random.Generator(np.random.Philox(21))
    lens = [3, 5, 20, 55]   # 1 x 128 tiles of these leave no room for the trial records
    chains = [inputs.random_saw(n, 1.0, rng) for n in lens]
    return inputs.System("chains", np.array(lens, np.int32), np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens]),
                         40.0, k_tors=-0.5, e_min=-400.0, bin_width=0.5, n_bins=1600, p=(0.3, 0.2, 0.3, 0.2), recompute_every=3,
                         walkers=walkers, xyz0=inputs.place_chains(chains, 40.0, 1.0, rng))


@pytest.mark.parametrize("kind,precision,walkers", [("sphere", 32, 1), ("sphere", 32, 153), ("sphere", 32, 20000), ("sphere", 64, 153),
                                                    ("chains", 32, 33), ("chains", 32, 700), ("chains", 64, 33)])
def test_tiles_give_the_same_walkers(phast, orc, kind, precision, walkers):
    s = _system(kind, walkers)
    n_sweeps, n_trace = 3, min(walkers, 2)
    got = []
    # FP64 records of the chains: four warps of them need more shared memory than an SM has
    for warps in (1, 2, 4) if (kind, precision) != ("chains", 64) else (1, 2):
        ctx = phast.Context(s, pair_precision=precision)
        ctx.set_tile(1, 32 * warps)
        trace = ctx.trace_buffer(n_sweeps, n_trace)
        hist = ctx.hist_sum_zeros()
        ctx.sweep(n_sweeps, ctx.lnW_zeros(), hist_sum=hist, trace=trace, trace_walkers=n_trace)
        st = ctx.get_state("cpu")
        torch.cuda.synchronize()
        got.append((st, hist.cpu(), trace.cpu().numpy().view(phast.TRACE_DTYPE).reshape(n_trace, -1)))
        ctx.close()
    st, hist, tr = got[0]
    for other, h, t in got[1:]:
        assert all(torch.equal(st[k], other[k]) for k in st), kind
        assert torch.equal(hist, h) and np.array_equal(tr["accepted"], t["accepted"])
    assert int(hist.sum()) == walkers * n_sweeps * s.n_total
    m, mu = oracle_model(orc, s), oracle_muca(orc, s)
    xyz = st["xyz"].numpy().reshape(walkers, s.n_total, 3)
    for w in range(n_trace):
        wk = orc.new_walker(m, mu, s.xyz0, int(s.seeds()[w]))
        force = None if precision == 64 else tr[w]["accepted"].astype(np.uint8)
        orc.sweep_walker(m, mu, np.zeros(s.n_bins), wk, n_sweeps * s.n_total, **({} if force is None else {"force": force}))
        assert np.array_equal(xyz[w], wk.xyz), (kind, precision, w)
