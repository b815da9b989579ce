"""FP32 tiles of 8 and 16 lanes per walker that run on a warp per walker (few walkers): the same trajectories, bit for bit, as
the groups of 8 and 16 lanes that many walkers get (one to three rounds of partners, partners beyond the last, all builds)."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1702_01770_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _system(kind):
    if kind == "sphere":
        return inputs.fene_sphere(1)
    lens = {"one": [3], "short": [9] * 4, "long": [3, 8, 17, 33, 5], "straight": [9, 21, 4]}[kind]
    rng = np.random.Generator(np.random.Philox(31))
    seq = np.concatenate([inputs.random_sequence(n, 0.5, rng) for n in lens])
    chains = [inputs.straight_chain(n) if kind == "straight" else inputs.random_saw(n, 1.0, rng) for n in lens]
    xyz0 = np.concatenate([c + np.array([0.0, 5.0 * i, 0.0]) for i, c in enumerate(chains)]) if kind == "straight" else \
        inputs.place_chains(chains, 40.0, 1.0, rng)
    return inputs.System(kind, np.array(lens, np.int32), seq, 0.0 if len(lens) == 1 else 40.0, k_tors=-0.5, e_min=-300.0, bin_width=0.25,
                         n_bins=2400, p=(0.3, 0.2, 0.3, 0.2), walkers=1, xyz0=xyz0)


@pytest.mark.parametrize("kind", ["one", "short", "long", "straight", "sphere"])
@pytest.mark.parametrize("tile", [(16, 2), (16, 32), (8, 16)])
def test_wide_groups_keep_the_tiles_trajectories(phast, kind, tile):
    n_sweeps, n_trace, out = 4, 4, []
    for walkers in (40, 3000, 5200):   # a warp each, a warp each on the 64-register build (16 lanes), the tile's groups
        s = dataclasses.replace(_system(kind), walkers=walkers, recompute_every=3)
        ctx = phast.Context(s, pair_precision=32)
        ctx.set_tile(*tile)
        trace = ctx.trace_buffer(n_sweeps, n_trace)
        hw = ctx.hist_walker_zeros()
        ctx.sweep(n_sweeps, ctx.lnW_zeros(), hist_walker=hw, trace=trace, trace_walkers=n_trace)
        st = ctx.get_state("cpu")
        torch.cuda.synchronize()
        N, K = s.n_total, s.n_bins
        out.append((st["xyz"][:40 * N * 3].numpy().copy(), st["E"][:40].numpy().copy(), st["bin"][:40].numpy().copy(),
                    hw[:40 * K].cpu().numpy(), trace.cpu().numpy().view(phast.TRACE_DTYPE).reshape(n_trace, -1)))
        ctx.close()
    for got in out[:2]:
        ref = out[2]
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[2], ref[2]) and np.array_equal(got[3], ref[3])
        assert np.all(np.abs(got[1] - ref[1]) <= 1e-11 * np.maximum(1.0, np.abs(ref[1])))   # FP64 recomputes: lane order
        assert np.array_equal(got[4]["accepted"], ref[4]["accepted"])
        if kind != "sphere":   # FENE changes in FP64 are summed in lane order
            assert np.array_equal(got[4]["dE"], ref[4]["dE"], equal_nan=True)
