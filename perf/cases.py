"""What is measured when the library is made faster: the work a user has it do, through the public entry points.

The kinds of work (``case["kind"]``):

* ``iteration``: one multicanonical iteration (clear the histograms, sweep every walker, Berg's weight step) replayed
  as the captured CUDA graph, as a production run does thousands of times in a row;
* ``sweep``: the same iteration as separate calls, as the short weight iterations of the small systems are run;
* ``energy``: energies of a batch of stored conformations, down to a single one;
* ``train``: one training step through autograd, coordinates and force-field parameters FP32 leaves;
* ``grad64``: energies and all derivatives in FP64 (the precision option of the derivative call);
* ``analyst``: the evaluation of a finished iteration: entropy, caloric curve and canonical averages with jackknife
  errors, then the free energy and the Maxwell construction;
* ``reweight``: canonical averages and their parameter derivatives from multicanonical samples on a temperature grid.

Sizes are those of the workloads in ``inputs.py`` and ``bench.py``.  FP32 sweeps have no 64-bit counterpart (a walker's
decisions follow from the FP32 energies), so ``exact`` gives values for them only in FP64 mode on a single open chain.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_1702_01770_gb300 import inputs, phast

KAPPA_C, KAPPA_LJ = 0.25, 4.0
C_LJ = (1.0, -0.5, -0.5, 0.5)          # AA, AB, BA, BB
MIX = (0.70, 0.15, 0.15, 0.0)
FIB = {13: "ABBABBABABBAB"}


# ---------------------------------------------------------------------------------------------------------------
# The cases.
# ---------------------------------------------------------------------------------------------------------------
def listed():
    return [
        # the large aggregation run: eight 55-mers, every walker of the full-size run, one sweep an iteration
        dict(name="iter_8x55", kind="iteration", system="8x55", walkers=16384, sweeps=1, blocks=16, precision=32, tile=""),
        # uneven system types sharing one launch (13-mer, 21-mer, two 34-mers, eight 9-mers), on the tile the autotuner picks
        dict(name="iter_uneven", kind="iteration", system="uneven", walkers=1024, sweeps=10, blocks=16, precision=32, tile="32x16"),
        # the paper's size class in a periodic box: four 9-mers, a few hundred walkers, a short weight iteration
        dict(name="sweep_4x9", kind="sweep", system="4x9", walkers=256, sweeps=10, blocks=1, precision=32, tile=""),
        # the smallest run: one 13-mer, eight walkers, all FP64 (latency of one walker's chain of moves)
        dict(name="sweep_13_f64", kind="sweep", system="13", walkers=8, sweeps=10, blocks=1, precision=64, tile=""),
        # the paper's own geometry (sphere, FENE bonds, six move types), one walker per thread as the autotuner picks
        dict(name="sweep_sphere", kind="sweep", system="sphere", walkers=16384, sweeps=10, blocks=1, precision=32, tile="1x128"),
        # FP64 energies of stored conformations of the large system (checking a run's running energies)
        dict(name="energy_8x55_f64", kind="energy", system="8x55", batch=1024, precision=64),
        # the energy of one conformation: call latency
        dict(name="energy_13_one", kind="energy", system="13", batch=1, precision=64),
        # force-field training on a batch of conformations of one 55-mer in open space
        dict(name="train_55", kind="train", system="55", batch=65536),
        # the same on several chains in a periodic box
        dict(name="train_8x9", kind="train", system="8x9", batch=8191),
        # all derivatives in FP64
        dict(name="grad_55_f64", kind="grad64", system="55", batch=4096),
        # evaluation of the large run: 8000 bins, 64 temperatures, 16 jackknife blocks
        dict(name="analyst_8000", kind="analyst", bins=8000, temps=64, blocks=16),
        # reweighted averages and sensitivities of 65536 samples at 64 temperatures
        dict(name="reweight_65536", kind="reweight", samples=65536, temps=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iteration", "sweep", "sweep64", "sphere", "energy", "train", "grad64", "analyst", "reweight"])
    if kind == "iteration":
        system = rng.choice(["8x55", "uneven", "2x34", "8x9"])
        walkers = _log(rng, 600, 16384) if system == "8x55" else _log(rng, 100, 2000)
        sweeps = 1 if system == "8x55" else rng.randint(2, 10)
        return dict(kind="iteration", system=system, walkers=walkers, sweeps=sweeps, blocks=rng.choice([1, 7, 16]), precision=32,
                    tile="" if system == "8x55" else rng.choice(["", "32x16", "32x8"]))
    if kind == "sweep":
        return dict(kind="sweep", system=rng.choice(["4x9", "13", "21"]), walkers=_log(rng, 60, 4000), sweeps=rng.randint(2, 20),
                    blocks=rng.choice([1, 5]), precision=32, tile=rng.choice(["", "32x4"]))
    if kind == "sweep64":
        return dict(kind="sweep", system=rng.choice(["13", "21", "4x9", "2x34"]), walkers=_log(rng, 4, 300), sweeps=rng.randint(1, 12),
                    blocks=rng.choice([1, 3]), precision=64, tile="")
    if kind == "sphere":
        return dict(kind="sweep", system="sphere", walkers=_log(rng, 1000, 65536), sweeps=rng.randint(2, 10), blocks=rng.choice([1, 16]),
                    precision=32, tile=rng.choice(["", "1x32", "1x64", "1x128"]))
    if kind == "energy":
        system = rng.choice(["13", "4x9", "55", "8x55"])
        return dict(kind="energy", system=system, batch=_log(rng, 1, {"13": 65536, "4x9": 32768, "55": 16384, "8x55": 1024}[system]),
                    precision=rng.choice([32, 64]))
    if kind == "train":
        system = rng.choice(["13", "21", "55", "4x9", "8x9", "2x34"])
        return dict(kind="train", system=system, batch=_log(rng, 200, {"13": 65536, "21": 65536, "55": 65536}.get(system, 16384)))
    if kind == "grad64":
        return dict(kind="grad64", system=rng.choice(["13", "21", "55", "4x9", "8x9"]), batch=_log(rng, 60, 8192))
    if kind == "analyst":
        return dict(kind="analyst", bins=_log(rng, 200, 16384), temps=rng.randint(8, 128), blocks=rng.choice([1, 2, 5, 16, 32]))
    return dict(kind="reweight", samples=_log(rng, 1000, 200000), temps=rng.randint(8, 128))


# ---------------------------------------------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------------------------------------------
def _seq(name, seed):
    """(chain lengths, sequence, box side, torsion weight) of a system; random sequences from the seed."""
    rng = np.random.default_rng(seed)
    if name in ("13", "21", "55"):
        n = int(name)
        return [n], inputs.fibonacci_sequence(n), 0.0, 0.0 if n == 13 else -0.5
    nc, n, frac, L = {"4x9": (4, 9, 0.5, 20.0), "8x9": (8, 9, 0.4, 30.0), "2x34": (2, 34, 0.4, 40.0), "8x55": (8, 55, 0.45, 40.0)}[name]
    return [n] * nc, (rng.random(nc * n) >= frac).astype(np.uint8), L, -0.5


def _systems(case, seed):
    """The system types of a run, with starts and walker keys from the seed."""
    W, name = case["walkers"], case["system"]
    if name == "sphere":
        types = [inputs.fene_sphere(W, seed=seed % (1 << 31))]
    elif name == "uneven":
        types = inputs.config2(W)
    elif name == "13":
        types = [inputs.config0(W)]
        if case["precision"] == 32:   # the same chain with torsion, as in the uneven run
            types = [dataclasses.replace(inputs.config2(W)[0])]
    elif name == "21":
        types = [inputs.config2(W)[1]]
    elif name in ("2x34", "8x9"):
        types = [inputs.config2(W)[2 if name == "2x34" else 3]]
    else:
        types = [inputs.config1(W) if name == "4x9" else inputs.config4(W)]
    rng, key, out = np.random.default_rng(seed), (seed * 7919 + 1) << 20, []
    for s in types:
        if s.box_L > 0:   # another start (single chains start straight, as in the workloads)
            chains = [inputs.random_saw(int(n), 1.0, rng) for n in s.chain_len]
            s = dataclasses.replace(s, xyz0=inputs.place_chains(chains, s.box_L, 1.0, rng))
        out.append(dataclasses.replace(s, seed_base=key))
        key += s.walkers
    return out


def _walks(gen, B, n, d_min=0.8, tries=8):
    """B random walks of n monomers with unit bonds, non-bonded distances >= d_min wherever one of a few draws allows it."""
    x = torch.zeros(B, n, 3, dtype=torch.float64, device="cuda")
    rows = torch.arange(B, device="cuda")
    for i in range(1, n):
        v = torch.randn(B, tries, 3, dtype=torch.float64, device="cuda", generator=gen)
        cand = x[:, i - 1, None] + v / v.norm(dim=2, keepdim=True)
        if i >= 2:
            d = torch.cdist(cand, x[:, : i - 1]).amin(2)
            pick = torch.where((d >= d_min).any(1), (d >= d_min).to(torch.int8).argmax(1), d.argmax(1))
        else:
            pick = torch.zeros_like(rows)
        x[:, i] = cand[rows, pick]
    return x


def _conformations(name, lens, L, B, seed):
    """A batch of conformations as a run of the system leaves them: walks, the chains placed apart from one another."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if len(lens) == 1:
        return _walks(gen, B, lens[0]).contiguous()
    out, a = torch.empty(B, sum(lens), 3, dtype=torch.float64, device="cuda"), 0
    for n in lens:
        c = _walks(gen, B, n)
        c = c - c.mean(1, keepdim=True)
        todo = torch.arange(B, device="cuda")
        for _ in range(40):
            new = c[todo] + torch.rand(todo.numel(), 1, 3, dtype=torch.float64, device="cuda", generator=gen) * L
            out[todo, a: a + n] = new
            if a == 0:
                break
            bad = []
            for part in todo.split(512):
                d = out[part, a: a + n, None] - out[part, None, :a]
                d = d - L * torch.round(d / L)
                bad.append(part[d.square().sum(3).amin((1, 2)) < 0.64])
            todo = torch.cat(bad)
            if todo.numel() == 0:
                break
        a += n
    return out.contiguous()


def _system_of(name, seed):
    lens, seq, L, kt = _seq(name, seed)
    return inputs.System(name, np.array(lens, np.int32), seq, L, k_tors=kt)


def _targets(B, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    return 20.0 * torch.randn(B, device="cuda", generator=gen)


def _entropy_run(case, seed):
    """Weights and block histograms of a nearly flat iteration over a transition: S(E) with a convex stretch, its ends
    rarely or never visited."""
    K, nb = case["bins"], case["blocks"]
    rng = np.random.default_rng(seed)
    w = 800.0 / 8000 if K > 2000 else 0.05
    e_min, N = -0.45 * K * w, 440 if K > 2000 else 36
    E = e_min + (np.arange(K) + 0.5) * w
    span, mid = K * w, e_min + 0.4 * K * w
    u = (E - e_min) / span
    S = N * (3.0 * np.log(u + 0.02) - 1.5 * u - 0.15 * np.exp(-(((E - mid) / (0.08 * span)) ** 2)))
    S -= S.max()
    flat = 0.15 * np.sin(9.0 * u + rng.uniform(0, 6.0)) + 0.05 * np.cumsum(rng.normal(size=K)) / math.sqrt(K)
    lam = 3000.0 * np.exp(flat) * (u > 0.01) * (u < 0.97)
    lam *= np.clip((u - 0.01) / 0.02, 0.0, 1.0)
    hist = rng.poisson(lam, size=(nb, K)).astype(np.int64)
    lnW = -S + flat
    lnW -= lnW[0]
    beta = np.gradient(S, E)
    T = np.linspace(0.6 / np.median(beta[K // 5: 3 * K // 4]), 2.0 / np.median(beta[K // 5: 3 * K // 4]), case["temps"])
    return lnW, hist, e_min, w, N, T


def _samples(case, seed):
    """Energies, their derivatives in one parameter and sampling log-weights of n states of a flat run, on the CPU."""
    gen = torch.Generator().manual_seed(seed)
    n = case["samples"]
    E = -60.0 + 160.0 * torch.rand(n, dtype=torch.float64, generator=gen)
    D = -0.4 * E + 5.0 * torch.randn(n, dtype=torch.float64, generator=gen) - 20.0
    u = (E + 65.0) / 170.0
    lnW = -(55.0 * (3.0 * torch.log(u) - 1.5 * u))
    return E, D, lnW, torch.linspace(0.1, 1.0, case["temps"], dtype=torch.float64)


# ---------------------------------------------------------------------------------------------------------------
# A pass.
# ---------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("iteration", "sweep"):
        types = _systems(case, seed)
        ctx = phast.Context(types, pair_precision=case["precision"])
        if case["tile"]:   # threads per walker x walkers per CTA, where it is not the default
            ctx.set_tile(*[int(v) for v in case["tile"].split("x")])
        st = dict(case=case, ctx=ctx, types=types, lnW=ctx.lnW_zeros(), hist=ctx.hist_sum_zeros(case["blocks"]))
        st["g_acc"] = torch.zeros_like(st["lnW"])
        if kind == "iteration":
            st["graph"] = ctx.capture_iteration(case["sweeps"], st["lnW"], st["hist"], st["g_acc"], n_jk=case["blocks"])
        return st
    if kind in ("energy", "train", "grad64"):
        s = _system_of(case["system"], seed)
        x = _conformations(case["system"], [int(n) for n in s.chain_len], s.box_L, case["batch"], seed)
        st = dict(case=case, system=s, x=x)
        if kind == "train":
            st["x"] = x.to(torch.float32).requires_grad_()
            st["params"] = torch.tensor(phast.ff_params(s), dtype=torch.float32, device="cuda", requires_grad=True)
            st["target"] = _targets(case["batch"], seed)
        return st
    if kind == "analyst":
        lnW, hist, e_min, w, N, T = _entropy_run(case, seed)
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        return dict(case=case, lnW=dev(lnW), hist=dev(hist), e_min=e_min, w=w, N=N, T=dev(T))
    E, D, lnW, T = _samples(case, seed)
    return dict(case=case, E=E.cuda(), D=D.cuda(), lnW=lnW.cuda(), T=T.cuda())


def _walkers(st):
    """What a program reads after an iteration: the weights, the histograms, the walkers and their counters."""
    s = st["ctx"].get_state()
    counters = s["stats"].view(torch.int64).view(-1, 18)[:, :15]   # attempts, accepts, pair evaluations, recomputes
    return dict(hist=st["hist"], lnW=st["lnW"], g_acc=st["g_acc"], xyz=s["xyz"], E=s["E"], bin=s["bin"], t=s["t"], counters=counters)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "iteration":
        state["graph"].launch()
        return _walkers(state)
    if kind == "sweep":
        s, nb = state["types"][0], case["blocks"]
        state["hist"].zero_()
        state["ctx"].sweep(case["sweeps"], state["lnW"], n_jk=nb, hist_sum=state["hist"])
        phast.phast_weight_update(state["hist"].view(nb, s.n_bins), state["lnW"], state["g_acc"], s.bin_width)
        return _walkers(state)
    if kind == "energy":
        return phast.phast_energy(state["system"], state["x"], pair_precision=case["precision"])
    if kind == "train":
        x, p = state["x"], state["params"]
        x.grad = p.grad = None
        loss = (phast.energy(x, p, state["system"]).float() - state["target"]).square().mean()
        loss.backward()
        return dict(loss=loss.detach(), grad_x=x.grad, grad_params=p.grad)
    if kind == "grad64":
        E, gx, gp = phast.phast_energy_grad(state["system"], state["x"], pair_precision=64)
        return dict(E=E, grad_x=gx, grad_params=gp)
    if kind == "analyst":
        a = (state["lnW"], state["e_min"], state["w"])
        r = phast.phast_micro_analysis(*a, hist=state["hist"], fd_half_width=5, n_monomers=state["N"], T=state["T"])
        f, rep, err = phast.phast_maxwell(state["lnW"], state["hist"], state["e_min"], state["w"], state["N"], fd_half_width=5)
        out = {k: v for k, v in vars(r).items() if v is not None}
        return dict(out, f=f, rep=rep, err=err)
    return phast.reweight_sensitivity(state["E"], state["D"], state["lnW"], 55, state["T"])


# ---------------------------------------------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------------------------------------------
def _sweep_pairs(s):
    """Expected pair evaluations of one move (inside a chain, between chains)."""
    n_in = n_out = 0.0
    N = s.n_total
    p = list(s.p) + [0.0] * (6 - len(s.p))
    for n in [int(v) for v in s.chain_len]:
        sides = [min(k, n - 1 - k) for k in range(1, n - 1)]
        piv_in = sum(2.0 * m * (n - m - 1) for m in sides) / len(sides)
        piv_out = sum(2.0 * m * (N - n) for m in sides) / len(sides)
        bonds = [min(l + 1, n - 1 - l) for l in range(n - 1)]
        bond_in = sum(2.0 * (m * (n - m) - 1) for m in bonds) / len(bonds)
        bond_out = sum(2.0 * m * (N - n) for m in bonds) / len(bonds)
        n_in += (p[0] * piv_in + p[3] * 2.0 * (n - 3) + p[4] * bond_in + p[5] * 2.0 * (n - 3)) / len(s.chain_len)
        n_out += (p[0] * piv_out + (p[1] + p[2]) * 2.0 * n * (N - n) + (p[3] + p[5]) * 2.0 * (N - n) + p[4] * bond_out) / len(s.chain_len)
    return n_in, n_out


def work(case):
    kind = case["kind"]
    if kind in ("iteration", "sweep"):
        W, bytes_, flops = case["walkers"], 0.0, 0.0
        for s in _types_for_work(case):
            n_in, n_out = _sweep_pairs(s)
            flops += W * s.n_total * case["sweeps"] * (14.0 * n_in + (23.0 if s.box_L > 0 else 14.0) * n_out)
            bytes_ += W * (2 * 24 * s.n_total + 2 * 20 + 8 + 2 * 144) + 8 * s.n_bins * (case["blocks"] + 4)
        return dict(bytes=bytes_, flops=flops)
    if kind in ("energy", "train", "grad64"):
        lens, _, L, _ = _seq(case["system"], 0)
        N, B = sum(lens), case["batch"]
        inter = sum(a * b for i, a in enumerate(lens) for b in lens[:i])
        intra = sum((n - 1) * (n - 2) / 2.0 for n in lens)
        per = 14.0 * intra + 23.0 * inter + 60.0 * N
        if kind == "energy":
            return dict(bytes=8.0 * B * (3 * N + 1), flops=B * per)
        per += 10.0 * (intra + inter) + 120.0 * N
        if kind == "train":
            return dict(bytes=B * (2 * 12.0 * N + 4), flops=B * per)
        return dict(bytes=8.0 * B * (6 * N + 6), flops=B * per)
    if kind == "analyst":
        K, nb, nT = case["bins"], case["blocks"], case["temps"]
        R = 1 + (nb if nb >= 2 else 0)
        return dict(bytes=8.0 * K * (1 + nb) * 2 + 8.0 * K * 7, flops=float(R) * K * (2 * nb + 60 + 40.0 * nT))
    return dict(bytes=8.0 * 3 * case["samples"], flops=40.0 * case["samples"] * case["temps"])


def _types_for_work(case):
    name = case["system"]
    one = {"sphere": inputs.fene_sphere, "13": inputs.config0, "4x9": inputs.config1, "8x55": inputs.config4}
    if name in one:
        return [one[name](case["walkers"])]
    t = inputs.config2(case["walkers"])
    return t if name == "uneven" else [t[{"21": 1, "2x34": 2, "8x9": 3}[name]]]


# ---------------------------------------------------------------------------------------------------------------
# The same results in 64 bits, by plain torch and numpy.
# ---------------------------------------------------------------------------------------------------------------
def _energy64(x, lens, seq, L, params):
    """Energies of x [B, N, 3] (FP64) under params (C_AA, C_BB, C_AB, kappa, kappa_C), differentiable."""
    N = x.shape[1]
    chain = torch.repeat_interleave(torch.arange(len(lens), device=x.device), torch.tensor(lens, device=x.device))
    i, j = torch.triu_indices(N, N, 1, device=x.device)
    inter = chain[i] != chain[j]
    keep = inter | (j - i >= 2)
    i, j, inter = i[keep], j[keep], inter[keep]
    s = torch.as_tensor(seq, device=x.device).long()
    c = params[torch.where(s[i] != s[j], 2, s[i])]
    d = x[:, i] - x[:, j]
    if L > 0:
        d = d - L * torch.round(d.detach() / L) * inter[None, :, None]
    r6 = d.square().sum(2) ** -3
    E = KAPPA_LJ * (r6 * (r6 - c)).sum(1)
    a = 0
    for n in lens:
        b = x[:, a + 1: a + n] - x[:, a: a + n - 1]
        u = b / b.norm(dim=2, keepdim=True)
        E = E + params[4] * (1.0 - (u[:, 1:] * u[:, :-1]).sum(2)).sum(1)
        if n >= 4:
            m = torch.linalg.cross(b[:, :-1], b[:, 1:])
            m = m / m.norm(dim=2, keepdim=True)
            E = E - params[3] * (m[:, 1:] * m[:, :-1]).sum(2).sum(1)
        a += n
    return E


def _exact_energy(case, seed):
    lens, seq, L, kt = _seq(case["system"], seed)
    x = _conformations(case["system"], lens, L, case["batch"], seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    p0 = torch.tensor([C_LJ[0], C_LJ[3], C_LJ[1], kt, KAPPA_C], **f64)
    N, kind = sum(lens), case["kind"]
    x = x.to(torch.float32).to(torch.float64) if kind == "train" else x
    step = max(1, int(4e6 // (N * N)))
    if kind == "energy":
        return torch.cat([_energy64(v, lens, seq, L, p0) for v in x.split(step)])
    E, gx, gp, loss, g_params = [], [], [], 0.0, torch.zeros(5, **f64)
    target = _targets(case["batch"], seed).double().split(step) if kind == "train" else None
    for k, v in enumerate(x.split(step)):
        v = v.clone().requires_grad_()
        if kind == "train":
            p = p0.clone().requires_grad_()
            part = (_energy64(v, lens, seq, L, p) - target[k]).square().sum() / case["batch"]
            a, b = torch.autograd.grad(part, (v, p))
            loss, g_params = loss + part.detach(), g_params + b
            gx.append(a)
        else:   # a row of parameters for each conformation gives each its own derivatives
            p = p0.expand(v.shape[0], 5).clone().requires_grad_()
            e = torch.func.vmap(lambda y, q: _energy64(y[None], lens, seq, L, q)[0])(v, p)
            a, b = torch.autograd.grad(e.sum(), (v, p))
            E.append(e.detach())
            gx.append(a)
            gp.append(b)
    if kind == "train":
        return dict(loss=loss, grad_x=torch.cat(gx), grad_params=g_params)
    return dict(E=torch.cat(E), grad_x=torch.cat(gx), grad_params=torch.cat(gp))


def _philox(c, key):
    """Philox4x32-10 of counters c (four uint64 arrays below 2^32) under 64-bit keys."""
    m = np.uint64(0xFFFFFFFF)
    k0, k1 = key & m, key >> np.uint64(32)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
    return c


def _exact_pivots(case, seed):
    """FP64 sweeps of one open chain under pivot moves, all walkers side by side."""
    s = _systems(case, seed)[0]
    n, W, K, w = s.n_total, case["walkers"], s.n_bins, s.bin_width
    iu, ju = np.triu_indices(n, 2)
    C = np.array(C_LJ)[2 * s.seq[iu].astype(int) + s.seq[ju]]
    key = (np.uint64(s.seed_base) + np.arange(W, dtype=np.uint64)).astype(np.uint64)

    def energy(x):
        r6 = ((x[:, iu] - x[:, ju]) ** 2).sum(2) ** -3.0
        e = KAPPA_LJ * (r6 * (r6 - C)).sum(1)
        b = np.diff(x, axis=1)
        u = b / np.linalg.norm(b, axis=2, keepdims=True)
        e = e + KAPPA_C * (1.0 - (u[:, 1:] * u[:, :-1]).sum(2)).sum(1)
        if s.k_tors != 0.0:
            m = np.cross(b[:, :-1], b[:, 1:])
            q = (m ** 2).sum(2)
            den = q[:, 1:] * q[:, :-1]
            cs = (m[:, 1:] * m[:, :-1]).sum(2) / np.sqrt(np.where(den < 1e-20, 1.0, den))
            e = e - s.k_tors * np.where(den < 1e-20, 0.0, cs).sum(1)
        return e

    def uniform(a, b):   # ((a >> 6) 2^26 + (b >> 6) + 1/2) 2^-52
        return ((a >> np.uint64(6)).astype(float) * 2.0 ** 26 + (b >> np.uint64(6)).astype(float) + 0.5) * 2.0 ** -52

    def block(t, b):
        z = np.zeros(W, np.uint64)
        return _philox([z + np.uint64(t), z, z + np.uint64(b), z + np.uint64(0x4D554341)], key)

    x = np.repeat(s.xyz0[None], W, 0)
    E = energy(x)
    bins = np.floor((E - s.e_min) / w).astype(int)
    hist = np.zeros((W, K))
    for t in range(case["sweeps"] * n):
        b0, b1, b2 = block(t, 0), block(t, 1), block(t, 2)
        idx = 1 + ((b0[3] * np.uint64(n - 2)) >> np.uint64(32)).astype(int)
        ang = (2.0 * uniform(b1[0], b1[1]) - 1.0) * s.amax[0]
        axis, won = np.tile([0.0, 0.0, 1.0], (W, 1)), np.zeros(W, bool)
        for j in range(64):
            b = block(t, 3 + j)
            v1, v2 = 2.0 * uniform(b[0], b[1]) - 1.0, 2.0 * uniform(b[2], b[3]) - 1.0
            q = v1 * v1 + v2 * v2
            new = ~won & (q < 1.0) & (q > 0.0)
            r = np.sqrt(np.where(new, 1.0 - q, 0.0))
            axis[new] = np.stack([2 * v1 * r, 2 * v2 * r, 1 - 2 * q], 1)[new]
            won |= new
            if won.all():
                break
        c = x[np.arange(W), idx]
        v = x - c[:, None]
        cs, sn = np.cos(ang)[:, None, None], np.sin(ang)[:, None, None]
        k = axis[:, None]
        rot = c[:, None] + v * cs + np.cross(np.broadcast_to(k, v.shape), v) * sn + k * (v * k).sum(2, keepdims=True) * (1 - cs)
        at = np.arange(n)[None]
        moved = np.where((idx < n - 1 - idx)[:, None], at < idx[:, None], at > idx[:, None])
        y = np.where(moved[:, :, None], rot, x)
        Ey = energy(y)
        by = np.floor((Ey - s.e_min) / w)
        ok = np.isfinite(Ey) & (by >= 0) & (by < K)   # the first iteration's weights are flat: in range is accepted
        x = np.where(ok[:, None, None], y, x)
        E = np.where(ok, Ey, E)
        bins = np.where(ok, by, bins).astype(int)
        hist[np.arange(W), bins] += 1
    H = hist.sum(0)
    both = (H[:-1] > 0) & (H[1:] > 0)
    h0, h1 = np.where(both, H[:-1], 1.0), np.where(both, H[1:], 1.0)
    g = np.where(both, h0 * h1 / (h0 + h1), 0.0)
    lnW = np.concatenate([[0.0], -np.cumsum(np.where(both, np.log(h1) - np.log(h0), 0.0))])
    return dict(hist=None, lnW=lnW, g_acc=np.concatenate([g, [0.0]]), xyz=x.reshape(-1), E=E, bin=None, t=None, counters=None)


def _exact_analyst(case, seed):
    lnW, hist, e_min, w, N, T = _entropy_run(case, seed)
    K, nb, h = case["bins"], case["blocks"], 5
    Ek = e_min + (np.arange(K) + 0.5) * w
    reps = [hist.sum(0)] + ([hist.sum(0) - hist[b] for b in range(nb)] if nb >= 2 else [])
    rows, mx = [], []
    for H in reps:
        with np.errstate(divide="ignore", invalid="ignore"):
            S = np.where(H > 0, -lnW + np.log(np.where(H > 0, H, 1)), np.nan)
            S = S - np.nanmax(S)
            beta, CV = np.full(K, np.nan), np.full(K, np.nan)
            beta[h:-h] = (S[2 * h:] - S[:-2 * h]) / (2 * h * w)
            s2 = (S[2 * h:] - 2 * S[h:-h] + S[:-2 * h]) / (h * w) ** 2
            CV[h:-h] = -(beta[h:-h] ** 2) / s2
            ok = ~np.isnan(S)
            a = S[ok][None] - Ek[ok][None] / T[:, None]
            p = np.exp(a - a.max(1, keepdims=True))
        Z = p.sum(1)
        m = (p * Ek[ok]).sum(1) / Z
        cv = (p * (Ek[ok][None] - m[:, None]) ** 2).sum(1) / Z / (N * T ** 2)
        i = int(np.argmax(cv))
        pk = [T[i], cv[i]]
        if 0 < i < len(T) - 1:
            x0, x1, x2, y0, y1, y2 = *T[i - 1: i + 2], *cv[i - 1: i + 2]
            num = (x1 - x0) ** 2 * (y1 - y2) - (x1 - x2) ** 2 * (y1 - y0)
            den = (x1 - x0) * (y1 - y2) - (x1 - x2) * (y1 - y0)
            xs = x1 - 0.5 * num / den
            pk = [xs, y0 * (xs - x1) * (xs - x2) / ((x0 - x1) * (x0 - x2)) + y1 * (xs - x0) * (xs - x2) / ((x1 - x0) * (x1 - x2))
                  + y2 * (xs - x0) * (xs - x1) / ((x2 - x0) * (x2 - x1))]
        rows.append((S, beta, CV, m, cv, np.array(pk)))
        mx.append(_maxwell(S, Ek, w, N, h))
    out = dict(zip(("S", "beta", "CV", "E_T", "cV_T", "peak"), rows[0]))
    bc = mx[0][0]
    out["f"] = (Ek - rows[0][0] / bc) / N if bc > 0 else np.full(K, np.nan)
    out["rep"], out["err"] = np.array(mx), np.full(6, np.nan)
    if nb >= 2:
        jk = lambda v: np.sqrt((nb - 1) / nb * ((v - v.mean(0)) ** 2).sum(0))  # noqa: E731
        for q, k in enumerate(("S", "beta", "CV", "E_T", "cV_T", "peak")):
            out[k + "_err"] = jk(np.array([r[q] for r in rows[1:]]))
        v = np.array(mx)[1:]
        if (v[:, 5] > 0).all():
            out["err"][:5] = jk(v[:, :5])
        out["err"][5] = (v[:, 5] > 0).sum()
    else:
        out["err"][5] = 0.0
    return out


def _maxwell(S, Ek, w, N, h):
    """The widest edge of the upper concave hull of S that spans visited bins and rises: (beta_c, eps_1, eps_2, latent
    heat, barrier, found)."""
    ks = np.nonzero(np.isfinite(S))[0]
    hull = []
    for k in ks:
        while len(hull) >= 2:
            i, j = hull[-2], hull[-1]
            if (S[j] - S[i]) * (Ek[k] - Ek[i]) <= (S[k] - S[i]) * (Ek[j] - Ek[i]):
                hull.pop()
            else:
                break
        hull.append(k)
    best = None
    for a, b in zip(hull[:-1], hull[1:]):
        if b - a < 2 or not np.isfinite(S[a + 1: b]).any() or not S[b] > S[a]:
            continue
        j = np.arange(max(a, h), min(b, len(S) - 1 - h) + 1)
        bk = S[j + h] - S[j - h]
        bk = bk[np.isfinite(bk)] / (2 * h * w)
        rise = np.max(bk - np.minimum.accumulate(bk)) if bk.size else 0.0
        if rise >= 0.0 and (best is None or Ek[b] - Ek[a] > best[0]):
            best = (Ek[b] - Ek[a], a, b)
    if best is None:
        return [np.nan] * 5 + [0.0]
    _, a, b = best
    bc = (S[b] - S[a]) / (Ek[b] - Ek[a])
    gap = np.nanmax(S[a] + bc * (Ek[a: b + 1] - Ek[a]) - S[a: b + 1])
    return [bc, Ek[a] / N, Ek[b] / N, (Ek[b] - Ek[a]) / N, gap / (bc * N), 1.0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("iteration", "sweep"):
        one = kind == "sweep" and case["precision"] == 64 and case["system"] in ("13", "21")
        return _exact_pivots(case, seed) if one else None
    if kind in ("energy", "train", "grad64"):
        return _exact_energy(case, seed)
    if kind == "analyst":
        return _exact_analyst(case, seed)
    E, D, lnW, T = _samples(case, seed)
    out = dict(E_T=[], cV_T=[], dE_T=[], dcV_T=[])
    for t in T:
        a = -E / t - lnW
        p = torch.exp(a - a.max())
        p = p / p.sum()
        e, d = E - (p * E).sum(), D - (p * D).sum()
        out["E_T"].append((p * E).sum())
        out["cV_T"].append((p * e * e).sum() / (55 * t * t))
        out["dE_T"].append((p * D).sum() - (p * e * d).sum() / t)
        out["dcV_T"].append((2.0 * (p * e * d).sum() - (p * e * e * d).sum() / t) / (55 * t * t))
    return {k: torch.stack(v) for k, v in out.items()}
