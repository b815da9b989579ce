"""A walker's results do not depend on how many others share its context: FP32 tiles of 8 and 16 lanes run on a warp per walker
while few walkers are there and on the tile's own groups when many are, and the FP64 sums (energy recomputes, exact local terms)
follow the tile's lane order in both, like the FP32 ones."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs

pytestmark = pytest.mark.gpu


def _system(kind):
    if kind == "4x9":
        return inputs.config1(1)
    if kind == "sphere":
        return inputs.fene_sphere(1)
    rng = np.random.Generator(np.random.Philox(31))
    lens = [3, 8, 17, 33, 5] if kind == "uneven" else [9, 21, 4]
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    chains = [inputs.straight_chain(n) if kind == "straight" else inputs.random_saw(n, 1.0, rng) for n in lens]
    xyz0 = np.concatenate([c + np.array([0.0, 5.0 * i, 0.0]) for i, c in enumerate(chains)]) if kind == "straight" else \
        inputs.place_chains(chains, 40.0, 1.0, rng)
    return inputs.System(kind, np.array(lens, np.int32), seq, 40.0, k_tors=-0.5, e_min=-300.0, bin_width=0.25, n_bins=2400,
                         p=(0.3, 0.2, 0.3, 0.2), walkers=1, xyz0=xyz0)


@pytest.mark.parametrize("kind", ["4x9", "uneven", "straight", "sphere"])
@pytest.mark.parametrize("tile", [(16, 2), (8, 16)])
def test_energies_of_few_and_many_walkers_are_the_same_bits(kind, tile):
    from paper_1702_01770_gb300 import phast
    n_sweeps, n_trace, out = 12, 8, []
    for walkers in (40, 3000, 5200):   # a warp each, (16 lanes) a warp each with 64 registers, the tile's groups
        s = dataclasses.replace(_system(kind), walkers=walkers, recompute_every=3)
        ctx = phast.Context(s, pair_precision=32)
        ctx.set_tile(*tile)
        trace = ctx.trace_buffer(n_sweeps, n_trace)
        ctx.sweep(n_sweeps, ctx.lnW_zeros(), trace=trace, trace_walkers=n_trace)
        st = ctx.get_state("cpu")
        torch.cuda.synchronize()
        tr = trace.cpu().numpy().view(phast.TRACE_DTYPE).reshape(n_trace, -1)
        out.append((st["xyz"][:40 * s.n_total * 3].numpy().copy(), st["E"][:40].numpy().copy(), tr["dE"].copy()))
        assert (ctx.stats()["recomputes"] == n_sweeps // 3).all()
        ctx.close()
    for got in out[:2]:
        for a, b in zip(got, out[2]):
            assert np.array_equal(a, b, equal_nan=True)
