"""The analysis kernels where their splits can go wrong: bins at and around the edges of CTAs and of what a CTA keeps,
few and many samples, temperatures whose weights underflow, hulls of smooth, noisy, gappy and exactly collinear
entropies, against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phast():
    from paper_1702_01770_gb300 import phast
    phast.lib()
    return phast


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _close(a, b, rtol, atol):
    a, b = np.asarray(a), np.asarray(b)
    assert np.array_equal(np.isnan(a), np.isnan(b))
    ok = ~np.isnan(a)
    assert np.all(np.abs(a[ok] - b[ok]) <= rtol * np.abs(b[ok]) + atol), np.max(np.abs(a[ok] - b[ok]))


@pytest.mark.parametrize("K", [3, 255, 256, 257, 513, 8192, 16384])
def test_micro_at_the_edges_of_its_ctas(phast, orc, K):
    """S, <E>_T and c_V(T) from the lowest temperatures, where all weights but a few underflow, to an infinite one.
    Tolerances: S to rounding of the logarithm and the shift; averages of exponentials of arguments up to |S|, |E/T|
    of some 10^4 carry 10^4 ulp each, 1e-11 relative."""
    rng = np.random.default_rng(K)
    e_min, w, h, N, nb = -0.3 * K * 0.1, 0.1, 1, 12, 3
    E = e_min + (np.arange(K) + 0.5) * w
    lnW = -40.0 * np.log(E - e_min + 1.0)
    H = rng.poisson(50.0, size=(nb, K)).astype(np.int64) + (K < 10)
    if K > 10:
        H[:, :2] = 0
        H[:, K // 3] = 0
    T = np.array([0.01, 0.05, 0.3, 1.0, 7.0, 1e6, np.inf])
    r = phast.phast_micro_analysis(_dev(lnW), e_min, w, hist=_dev(H), fd_half_width=h, n_monomers=N, T=_dev(T))
    o = orc.micro_analysis(lnW, e_min, w, H=H.sum(0).astype(float), fd_half_width=h, n_monomers=N, T=T)
    _close(r.S.cpu(), o["S"], 1e-13, 1e-12)
    _close(r.beta.cpu(), o["beta"], 1e-9, 1e-9)
    _close(r.E_T.cpu(), o["E_T"], 1e-11, 1e-11 * np.abs(E).max())
    _close(r.cV_T.cpu()[:-1], o["cV_T"][:-1], 1e-9, 1e-9)
    assert r.cV_T[-1].item() == 0.0
    reps = [orc.micro_analysis(lnW, e_min, w, H=(H.sum(0) - H[b]).astype(float), fd_half_width=h, n_monomers=N, T=T) for b in range(nb)]
    _close(r.E_T_err.cpu(), orc.jackknife([x["E_T"] for x in reps]), 1e-6, 1e-10 * np.abs(E).max())


@pytest.mark.parametrize("n", [1, 7, 8, 9, 2047, 8 * 6080, 8 * 6080 + 5, 200001])
def test_reweighting_of_few_and_many_samples(phast, orc, n):
    rng = np.random.default_rng(n)
    E, D, lnW = rng.uniform(-60, 100, n), rng.normal(0, 5, n), rng.uniform(-30, 0, n)
    T = np.array([0.05, 0.2, 0.9, 4.0])
    g = phast.reweight_sensitivity(_dev(E), _dev(D), _dev(lnW), 55, _dev(T))
    o = orc.reweight_sensitivity(E, D, lnW, 55, T)
    for k in ("E_T", "cV_T", "dE_T", "dcV_T"):   # sums of up to 2e5 terms in another order; moments of a few samples cancel
        scale = max(1.0, np.abs(o[k]).max())
        assert np.all(np.abs(g[k].cpu().numpy() - o[k]) <= 1e-10 * np.abs(o[k]) + 1e-11 * scale), (k, g[k].cpu().numpy(), o[k])


def _curves(K):
    x = np.linspace(0.0, 1.0, K)
    rng = np.random.default_rng(K)
    concave, bend = 60.0 * np.sqrt(x + 0.01), 60.0 * np.sqrt(x + 0.01) - 9.0 * np.exp(-((x - 0.4) / 0.1) ** 2)
    gaps = bend + 0.05 * rng.normal(size=K)
    gaps[rng.random(K) < 0.4] = np.nan
    gaps[: K // 20] = np.nan
    return {"concave": concave, "bend": bend, "noise": bend + 0.05 * rng.normal(size=K), "gaps": gaps, "flat": np.zeros(K),
            "line": 0.25 * np.arange(K), "pieces": np.minimum(0.5 * np.arange(K), 0.25 * np.arange(K) + K // 8),
            "convex": 30.0 * x * x, "steps": np.floor(8 * x) * 2.0 + 0.25 * (np.arange(K) % 2)}


@pytest.mark.parametrize("K", [4, 33, 511, 513, 2500])
@pytest.mark.parametrize("tol_beta", [0.0, 0.02])
def test_hulls_of_every_kind(phast, orc, K, tol_beta):
    """Row 0 elementwise against the oracle's sequential chain (values within rounding: the same vertices)."""
    e_min, w, N = -0.25 * K, 0.5, 20
    for name, S in _curves(K).items():
        lnW, H = -np.where(np.isnan(S), 0.0, S), (~np.isnan(S)).astype(np.int64)[None]
        f, rep, _ = phast.phast_maxwell(_dev(lnW), _dev(H), e_min, w, N, fd_half_width=1, tol_beta=tol_beta)
        Sn = np.where(H[0] > 0, -lnW, np.nan)
        fo, ro = orc.maxwell(Sn - np.nanmax(Sn), e_min, w, N, tol_beta=tol_beta)
        for q, key in enumerate(("beta_c", "eps_1", "eps_2", "latent", "barrier", "found")):
            got = rep[0, q].item()
            assert (np.isnan(got) and np.isnan(ro[key])) or abs(got - ro[key]) <= 1e-12 * max(1.0, abs(ro[key])), (name, key, got, ro[key])
        _close(f.cpu(), fo, 1e-13, 1e-12 * np.nanmax(np.abs(Sn - np.nanmax(Sn)), initial=1.0))


@pytest.mark.parametrize("types", [1, 3])
def test_weight_steps_of_a_captured_iteration(phast, orc, types):
    """Berg's step of every type of one launch, against the oracle's step on the iteration's own histograms."""
    from paper_1702_01770_gb300 import inputs
    systems = inputs.config2(walkers_each=6)[:types]
    ctx = phast.Context(systems, pair_precision=32)
    lnW, hist = ctx.lnW_zeros(), ctx.hist_sum_zeros(2)
    g, flat = torch.zeros_like(lnW), torch.zeros(types, 4, dtype=torch.float64, device="cuda")
    graph = ctx.capture_iteration(5, lnW, hist, g, n_jk=2, flat_out=flat)
    for _ in range(2):
        before, g0 = lnW.cpu().numpy().copy(), g.cpu().numpy().copy()
        graph.launch()
        torch.cuda.synchronize()
        off = 0
        for i, s in enumerate(systems):
            K, o = s.n_bins, ctx.lnw_off[i]
            H = hist[2 * off: 2 * (off + K)].view(2, K).sum(0).cpu().numpy().astype(float)
            ref, g_ref, f_ref = orc.berg_update(H, before[o: o + K], g0[o: o + K - 1], s.bin_width)
            assert np.allclose(lnW[o: o + K].cpu().numpy(), ref, rtol=0, atol=1e-9)
            assert np.allclose(g[o: o + K - 1].cpu().numpy(), g_ref, rtol=1e-12, atol=0)
            assert np.allclose(flat[i].cpu().numpy(), f_ref, rtol=1e-10)
            off += K
    ctx.close()


@pytest.mark.parametrize("n_blocks", [2, 6, 7, 13])
def test_replicates_far_from_the_full_histogram(phast, orc, n_blocks):
    """Blocks that visit disjoint energies: a replicate's mean then lies many of its own widths from the full
    histogram's, and at the lowest temperature all its weights underflow beside the full histogram's largest."""
    rng = np.random.default_rng(n_blocks)
    K, e_min, w, N = 1300, -50.0, 0.1, 9
    E = e_min + (np.arange(K) + 0.5) * w
    lnW = -0.3 * E
    H = np.zeros((n_blocks, K), np.int64)
    for b in range(n_blocks):
        lo = K * b // n_blocks
        H[b, lo: lo + 40] = rng.integers(1, 1000, 40)
    T = np.array([0.005, 0.1, 1.0, 3.0, 50.0])
    r = phast.phast_micro_analysis(_dev(lnW), e_min, w, hist=_dev(H), fd_half_width=2, n_monomers=N, T=_dev(T))
    o = orc.micro_analysis(lnW, e_min, w, H=H.sum(0).astype(float), fd_half_width=2, n_monomers=N, T=T)
    reps = [orc.micro_analysis(lnW, e_min, w, H=(H.sum(0) - H[b]).astype(float), fd_half_width=2, n_monomers=N, T=T) for b in range(n_blocks)]
    _close(r.E_T.cpu(), o["E_T"], 1e-11, 1e-9)
    _close(r.cV_T.cpu(), o["cV_T"], 1e-10, 1e-12)
    _close(r.E_T_err.cpu(), orc.jackknife([x["E_T"] for x in reps]), 1e-9, 1e-9)
    _close(r.cV_T_err.cpu(), orc.jackknife([x["cV_T"] for x in reps]), 1e-9, 1e-9)


@pytest.mark.parametrize("K,lo,hi", [(1, 0, 1), (2, 0, 2), (5, 0, 5), (9, 3, 4), (515, 0, 129), (2049, 600, 1500), (8001, 2000, 2001),
                                     (8001, 3990, 8001), (16384, 0, 16384)])
def test_maxwell_of_visits_in_one_stretch_of_the_bins(phast, orc, K, lo, hi):
    """The hull is put together from four stretches of the bins: visits confined to one or two of them, one visited bin, as few
    bins as stretches or fewer, and the largest size, a convex dip with noise each."""
    rng = np.random.default_rng(K + lo)
    x = np.linspace(-1.0, 1.0, K)
    S = 40.0 * (-x * x - 2.0 * np.exp(-((x - x[(lo + hi) // 2]) / 0.2) ** 2)) + 5.0 * x + 0.01 * rng.standard_normal(K)
    visited = (np.arange(K) >= lo) & (np.arange(K) < hi)
    lnW, H = -np.where(visited, S, 0.0), visited.astype(np.int64)[None]
    _, rep, _ = phast.phast_maxwell(_dev(lnW), _dev(H), -0.25 * K, 0.5, 20, fd_half_width=1)
    Sn = np.where(visited, -lnW, np.nan)
    _, ro = orc.maxwell(Sn - np.nanmax(Sn), -0.25 * K, 0.5, 20)
    for q, key in enumerate(("beta_c", "eps_1", "eps_2", "latent", "barrier", "found")):
        got = rep[0, q].item()
        assert (np.isnan(got) and np.isnan(ro[key])) or abs(got - ro[key]) <= 1e-12 * max(1.0, abs(ro[key])), (key, got, ro[key])
