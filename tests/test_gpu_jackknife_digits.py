"""Jackknife errors of <E>_T and c_V(T) to the last digits where a replicate's mean energy lies several of its spreads from the
full histogram's: two blocks of visits, one Gaussian in energy each."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gap", [0.2, 1.0, 3.0, 8.0, 14.0])   # centres 0.2 to 14 units apart, spreads 0.5 and 1
def test_replicates_some_spreads_apart(gap):
    """Against extended precision.  The error of two replicates is half their difference, c_V of the one about four times the
    other's: 24 roundings of 2^-53 (sums of a few bins a thread and a tree, the weights' exponentials and their arguments,
    variances about the mean) grow by (4 + 1) / (4 - 1); <E>'s likewise, relative to the energies themselves."""
    from paper_1702_01770_gb300 import phast
    K, w, e0, n_mono = 2000, 0.05, -50.0, 10
    LD = np.longdouble
    k = np.arange(K)
    e = e0 + (k + 0.5) * w
    h = np.stack([np.rint(1e9 * np.exp(-0.5 * ((e - c) / s) ** 2)) for c, s in ((-10.0, 0.5), (-10.0 + gap, 1.0))]).astype(np.int64)
    T = np.linspace(5.0, 50.0, 64)
    c = lambda a: torch.from_numpy(a).cuda()
    r = phast.phast_micro_analysis(c(np.zeros(K)), e0, w, c(h), n_monomers=n_mono, T=c(T))

    def canonical(H):
        H = H.astype(LD)
        E = LD(e0) + (k.astype(LD) + LD(0.5)) * LD(w)
        m = H > 0
        out = []
        for t in T.astype(LD):
            a = np.log(H[m]) - E[m] / t
            p = np.exp(a - a.max())
            mean = (p * E[m]).sum() / p.sum()
            out.append((mean, (p * (E[m] - mean) ** 2).sum() / p.sum() / (n_mono * t * t)))
        return np.array(out).T

    full, one, two = canonical(h.sum(0)), canonical(h[1]), canonical(h[0])
    tol = 24 * 2.0 ** -53 * 5 / 3
    for got, err, q in ((r.E_T, r.E_T_err, 0), (r.cV_T, r.cV_T_err, 1)):
        size = np.abs(full[q]) + np.abs(one[q]) + np.abs(two[q]) if q == 0 else np.abs(one[q] - two[q]) / 2
        assert np.all(np.abs(got.cpu().numpy() - full[q]) <= tol * np.abs(full[q]))
        assert np.all(np.abs(err.cpu().numpy() - np.abs(one[q] - two[q]) / 2) <= tol * size)


@pytest.mark.parametrize("blocks", [0, 1, 3])
@pytest.mark.parametrize("binned", [False, True])
def test_specific_heat_of_a_frozen_system(blocks, binned):
    """Temperatures so low that one bin has all the weight: c_V is that of the next one, exp(-dE / T) of it (1e-87 to 1e-9), to
    the rounding of the exponents (2^-53 of 40 / T each) and two dozen others."""
    from paper_1702_01770_gb300 import phast
    K, w, e0, n = 500, 0.1, -20.0, 9
    T = np.array([0.0005, 0.001, 0.002, 0.005])
    lnW = np.zeros(K)
    H = None if blocks == 0 else np.full((blocks, K), 7, np.int64)
    c = lambda a: None if a is None else torch.from_numpy(a).cuda()
    if binned:
        r = phast.phast_micro_analysis_binned(c(np.zeros((2, K))), e0, w, c(np.full((2, K), 7, np.int64)), block=1, n_monomers=n, T=c(T))
    else:
        r = phast.phast_micro_analysis(c(lnW), e0, w, c(H), n_monomers=n, T=c(T))
    LD = np.longdouble
    E = LD(e0) + (np.arange(K).astype(LD) + LD(0.5)) * LD(w)
    for t, got in zip(T, r.cV_T.cpu().numpy()):
        p = np.exp(-(E - E[0]) / LD(t))
        mean = (p * E).sum() / p.sum()
        ref = (p * (E - mean) ** 2).sum() / p.sum() / (n * LD(t) ** 2)
        assert abs(got - ref) <= 2.0 ** -53 * (4 * 40 / t + 24) * ref, (t, got, ref)
