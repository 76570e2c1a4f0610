"""The workloads that the library is timed on, as a user's program runs them.

Every case is one leg of a Monte Carlo program through the Python binding
(paper_2604_08250_gb300.smc): measure the configuration in hand (energy,
short-range order, gradient), then sweep it on by some sweeps, so that calling
run() again continues the chain.  The kinds are the package's named workloads
(inputs.CONFIG1 - CONFIG5 and the qSRO, MLPNet and FCC workloads of bench.py):

  small      BCC, integer pair model, a box of a few cells (also odd ones)
  anneal     BCC, FP32 pair model, the lattice fits the SMs' shared memory
  stream     BCC, FP32 pair model, lattices larger than that
  job        BCC, start configuration + sweeps + observables, up to 3 shells
             and 8 species, rows of any multiple of four cells
  ladder     BCC, replicas of uneven sizes on a temperature ladder, one call
  mlp        BCC, 20-64-64-1 SiLU network
  sample     BCC, pair + MLP model: SRO, dE/dtheta, one sweep (a sample of
             d<SRO>/dtheta)
  mlpnet     BCC, 20-96-96-96-1 ReLU network
  fit        BCC, E(theta) and its gradient through torch.autograd
  qsro       BCC, qSRO model
  fcc        FCC, FP32 or integer pair model
  fcc_qsro   FCC, qSRO model, Fe29Co29Ni28Al7Ti7
"""
from __future__ import annotations

import itertools

import numpy as np
import torch

from paper_2604_08250_gb300 import inputs, smc

K_B = inputs.K_B_EV
Z_BCC, Z_FCC = (8, 6, 12), (12, 6, 24)


def listed():
    return [
        # CONFIG1 as it stands: 8^3, two species, 100 sweeps at kT = 25 meV (latency of the smallest call)
        dict(name="small_8", kind="small", nx=8, ny=8, nz=8, S=2, shells=2, sweeps=100),
        # CONFIG2: 128^3 anneal 3000 -> 300 K; 100 of its 1000 temperatures per leg
        dict(name="anneal_128", kind="anneal", nx=128, ny=128, nz=128, S=5, shells=2, sweeps=100),
        # the largest lattice of the package (512^3, 268 M sites): a few sweeps and the pair gradient
        dict(name="stream_512", kind="stream", nx=512, ny=512, nz=512, S=5, shells=2, sweeps=4),
        # a whole short job on an uneven box: start state, 8 species, 3 shells, energy and SRO
        dict(name="job_200x120x88", kind="job", nx=200, ny=120, nz=88, S=8, shells=3, sweeps=10),
        # CONFIG3: 64 cubes of 36^3 - 96^3 cells, 300 - 3000 K, one call
        dict(name="ladder_64", kind="ladder", R=64, lo=8, hi=24, S=5, shells=2, sweeps=20),
        # CONFIG4: 256^3, Dirichlet composition, 800 K; 10 of its 200 sweeps
        dict(name="mlp_256", kind="mlp", nx=256, ny=256, nz=256, S=5, sweeps=10),
        # CONFIG5: 512^3, one sample at 600 K: SRO, dE/dtheta (5599 parameters), one sweep
        dict(name="sample_512", kind="sample", nx=512, ny=512, nz=512, S=5, shells=2, sweeps=1),
        # the paper's network on a middle-sized box
        dict(name="mlpnet_128", kind="mlpnet", nx=128, ny=128, nz=128, S=5, sweeps=10),
        # fitting interactions: energy and gradient of a small box through torch.autograd
        dict(name="fit_32", kind="fit", nx=32, ny=32, nz=32, S=5, shells=2),
        # qSRO workload, 256^3, 800 K
        dict(name="qsro_256", kind="qsro", nx=256, ny=256, nz=256, S=5, shells=2, sweeps=4),
        # the paper's lattice, 256^3 cubic cells (67 M sites), pair model, 800 K
        dict(name="fcc_256", kind="fcc", nx=256, ny=256, nz=256, S=5, shells=2, sweeps=2, integer=False),
        # the paper's lattice, model and alloy on a middle-sized box, 800 K
        dict(name="fcc_qsro_128", kind="fcc_qsro", nx=128, ny=128, nz=128, S=5, shells=2, sweeps=4),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _axes(rng, lo, hi, most, step=4):
    """Three axis lengths, multiples of `step`, their product at most `most`."""
    while True:
        d = [max(lo, _log(rng, lo, hi) // step * step) for _ in range(3)]
        if d[0] * d[1] * d[2] <= most:
            return dict(nx=d[0], ny=d[1], nz=d[2])


def draw(rng):
    kind = rng.choice(["small", "anneal", "stream", "job", "ladder", "mlp", "sample", "mlpnet", "fit", "qsro", "fcc",
                       "fcc_qsro"])
    if kind == "small":  # any box, also axes that are no multiple of four
        return dict(kind=kind, nx=rng.randint(4, 12), ny=rng.randint(4, 12), nz=rng.randint(4, 12),
                    S=rng.randint(2, 4), shells=rng.randint(1, 3), sweeps=rng.randint(2, 20))
    if kind == "anneal":
        d = _axes(rng, 16, 160, 128 ** 3)
        return dict(kind=kind, **d, S=rng.randint(2, 5), shells=2, sweeps=rng.randint(20, 200))
    if kind == "stream":
        d = _axes(rng, 128, 512, 512 ** 3)
        if rng.random() < 0.5:  # the row lengths that large boxes usually have
            d["nx"] = rng.choice([128, 256, 512])
        return dict(kind=kind, **d, S=5, shells=2, sweeps=rng.randint(1, 4))
    if kind == "job":
        d = _axes(rng, 16, 256, 200 * 120 * 88)
        return dict(kind=kind, **d, S=rng.randint(2, 8), shells=rng.randint(1, 3), sweeps=rng.randint(2, 10))
    if kind == "ladder":
        return dict(kind=kind, R=rng.randint(2, 64), lo=rng.randint(2, 8), hi=rng.randint(9, 24), S=5, shells=2,
                    sweeps=rng.randint(2, 20))
    if kind == "mlp":
        d = _axes(rng, 16, 256, 256 ** 3)
        return dict(kind=kind, **d, S=rng.randint(2, 5), sweeps=rng.randint(1, 10))
    if kind == "sample":
        d = _axes(rng, 16, 512, 512 ** 3)
        return dict(kind=kind, **d, S=rng.randint(3, 5), shells=rng.randint(1, 3), sweeps=1)
    if kind == "mlpnet":
        d = _axes(rng, 16, 256, 256 ** 3)
        n = d["nx"] * d["ny"] * d["nz"]
        return dict(kind=kind, **d, S=5, sweeps=rng.randint(1, 10) if n <= 128 ** 3 else 2)
    if kind == "fit":  # odd axes too: energies and gradients take any box
        return dict(kind=kind, nx=_log(rng, 6, 64), ny=_log(rng, 6, 64), nz=_log(rng, 6, 64), S=rng.randint(2, 5),
                    shells=rng.randint(1, 3))
    if kind == "qsro":
        d = _axes(rng, 16, 256, 256 ** 3)
        return dict(kind=kind, **d, S=rng.randint(2, 8), shells=rng.randint(1, 3), sweeps=rng.randint(1, 4))
    if kind == "fcc":
        d = _axes(rng, 8, 256, 256 ** 3)
        return dict(kind=kind, **d, S=rng.randint(2, 8), shells=rng.randint(1, 3), sweeps=rng.randint(1, 2),
                    integer=rng.random() < 0.3)
    d = _axes(rng, 8, 256, 128 ** 3)
    return dict(kind=kind, **d, S=5, shells=rng.randint(1, 3), sweeps=rng.randint(1, 4))


def _sites(c):
    per = 4 if c["kind"].startswith("fcc") else 2
    if c["kind"] == "ladder":
        return sum(2 * int(e) ** 3 for e in _edges(c))
    return per * c["nx"] * c["ny"] * c["nz"]


def _edges(c):
    return inputs.batched_edges(inputs.CONFIG3["edge_seed"], c["R"], c["lo"], c["hi"])


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _occupancy(n, fractions, seed):
    """A random alloy: n sites, species drawn with the given fractions."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    cum = torch.tensor(np.cumsum(np.asarray(fractions, dtype=np.float64))[:-1], dtype=torch.float32, device="cuda")
    out = torch.empty(n, dtype=torch.int8, device="cuda")
    step = 1 << 26
    for i in range(0, n, step):
        u = torch.rand(min(step, n - i), generator=g, device="cuda")
        out[i:i + step] = torch.bucketize(u, cum, out_int32=True, right=True).to(torch.int8)
    return out


def _fractions(c, seed):
    S = c["S"]
    if c["kind"] in ("mlp", "mlpnet", "qsro"):  # their workloads' Dirichlet compositions
        return np.random.default_rng(seed).dirichlet(np.full(S, 5.0))
    if c["kind"] == "fcc_qsro":
        return inputs.HEA_FRACTIONS
    return np.full(S, 1.0 / S)


def _parameters(c, seed):
    """Model parameters as arrays (host), by kind."""
    S, kind = c["S"], c["kind"]
    if kind == "small" or (kind == "fcc" and c["integer"]):
        return dict(v=inputs.pair_int_coeffs(seed, c["shells"], S))
    if kind in ("anneal", "stream", "job", "ladder", "fcc"):
        return dict(v=inputs.pair_f32_coeffs(seed, c["shells"], S))
    if kind in ("qsro", "fcc_qsro"):
        v, w, k = inputs.qsro_coeffs(seed, c["shells"], S)
        return dict(v=v, w=w, c=k)
    if kind == "mlp":
        return dict(mlp=inputs.mlp_weights(seed))
    if kind == "mlpnet":
        return dict(net=inputs.mlpnet_weights(seed))
    return dict(v=inputs.pair_f32_coeffs(seed, c["shells"], S), mlp=inputs.mlp_weights(seed))  # sample, fit


def _model(c, p):
    kind = c["kind"]
    if kind == "small" or (kind == "fcc" and c["integer"]):
        return smc.Model(smc.PAIR_I32, c["shells"], p["v"], unit_ev=1e-4)
    if kind in ("anneal", "stream", "job", "ladder", "fcc"):
        return smc.Model(smc.PAIR_F32, c["shells"], p["v"])
    if kind in ("qsro", "fcc_qsro"):
        return smc.Model(smc.QSRO_F32, c["shells"], p["v"], qsro_w=p["w"], qsro_c=p["c"])
    if kind == "mlp":
        return smc.Model(smc.MLP_BF16, mlp=p["mlp"])
    if kind == "mlpnet":
        return smc.Model(smc.MLPNET_BF16, net=p["net"])
    return smc.Model(smc.PAIR_F32_MLP_BF16, c["shells"], p["v"], mlp=p["mlp"])


def _theta(c, p):
    """The flat parameter vector of a pair + MLP model: V_m(p, q), p <= q, then W1, b1, W2, b2, W3, b3."""
    S = c["S"]
    up = np.triu_indices(S)
    m = p["mlp"]
    w = {k: inputs.bf16_bits_to_f32(m[k]) for k in ("w1", "w2", "w3")}
    parts = [p["v"][s][up] for s in range(c["shells"])] + [w["w1"], m["b1"], w["w2"], m["b2"], w["w3"], [m["b3"]]]
    return np.concatenate([np.asarray(x, dtype=np.float32).reshape(-1) for x in parts])


def prepare(case, seed):
    c = dict(case)
    p = _parameters(c, seed)
    st = dict(c=c, seed=seed, sweep=0)
    if c["kind"] == "fit":
        st["lat"] = smc.Lattice(c["nx"], c["ny"], c["nz"], c["S"])
        st["occ"] = _occupancy(st["lat"].nsites, _fractions(c, seed), seed)
        st["theta"] = torch.tensor(_theta(c, p), device="cuda", requires_grad=True)
        return st
    R = c.get("R", 1)
    st["model"] = _model(c, p)
    st["e_acc"] = torch.zeros(R, dtype=torch.float64, device="cuda")
    st["n_acc"] = torch.zeros(R, dtype=torch.int64, device="cuda")
    st["e"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    nsh = 3 if c["kind"] in ("anneal", "sample") else c.get("shells", 1)
    st["counts"] = torch.zeros((nsh, c["S"], c["S"]), dtype=torch.int64, device="cuda")
    st["alpha"] = torch.zeros((nsh, c["S"], c["S"]), dtype=torch.float64, device="cuda")
    n = c.get("sweeps", 0)
    if c["kind"] == "ladder":
        st["lats"] = [smc.Lattice(int(e), int(e), int(e), c["S"]) for e in _edges(c)]
        st["occ"] = _occupancy(_sites(c), _fractions(c, seed), seed)  # one buffer, a slice for each replica
        st["occs"] = list(torch.split(st["occ"], [l.nsites for l in st["lats"]]))
        st["kT"] = np.repeat(inputs.ladder_kT(R)[:, None], n, axis=1)
        return st
    st["lat"] = smc.Lattice(c["nx"], c["ny"], c["nz"], c["S"])
    if c["kind"] == "job":
        st["occ"] = torch.empty(st["lat"].nsites, dtype=torch.int8, device="cuda")
        st["start"] = inputs.equiatomic_counts(st["lat"].nsites, c["S"])
    else:
        st["occ"] = _occupancy(_sites(c), _fractions(c, seed), seed)
    if c["kind"] in ("stream", "sample"):
        st["grad"] = torch.zeros(smc.grad_size(st["lat"], st["model"]), dtype=torch.float32, device="cuda")
    st["e_int"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    if c["kind"] == "small":
        st["kT"] = inputs.CONFIG1["kT_ev"]
    elif c["kind"] in ("anneal", "job"):
        st["kT"] = inputs.anneal_kT(n)
    elif c["kind"] == "sample":
        st["kT"] = K_B * inputs.CONFIG5["T"]
    else:
        st["kT"] = K_B * 800.0
    return st


# ---------------------------------------------------------------------------
# One pass.
# ---------------------------------------------------------------------------
def run(st):
    c, kind = st["c"], st["c"]["kind"]
    if kind == "fit":
        lat, theta = st["lat"], st["theta"]
        theta.grad = None
        e = smc.smc_energy_fn(theta, lat, st["occ"], smc.PAIR_F32_MLP_BF16, c["shells"])
        e.backward()
        return {"e": e.detach(), "grad": theta.grad}
    n, s0, seed = c["sweeps"], st["sweep"], st["seed"]
    model, e, e_acc, n_acc = st["model"], st["e"], st["e_acc"], st["n_acc"]
    st["sweep"] = s0 + n
    out = {"e_acc": e_acc, "n_acc": n_acc}
    if kind == "ladder":
        smc.sweep_batched(st["lats"], model, st["occs"], seed, s0, n, st["kT"], e_acc=e_acc, n_acc=n_acc)
        out["occ"] = st["occ"]
        return out
    lat, occ = st["lat"], st["occ"]
    out["occ"] = occ
    if kind in ("fcc", "fcc_qsro"):
        if kind == "fcc" and c["integer"]:
            smc.fcc_energy(lat, model, occ, e, st["e_int"])
            out["e_int"] = st["e_int"]
        else:
            smc.fcc_energy(lat, model, occ, e)
        smc.fcc_sweep(lat, model, occ, seed, s0, n, st["kT"], e_acc=e_acc, n_acc=n_acc)
        out["e"] = e
        return out
    if kind == "small":
        smc.energy(lat, model, occ, e, st["e_int"])
        out.update(e=e, e_int=st["e_int"])
    elif kind == "job":
        smc.init_lattice(lat, st["start"], seed, occ)
    elif kind in ("anneal", "mlp", "mlpnet", "qsro"):
        smc.energy(lat, model, occ, e)
        out["e"] = e
    if kind in ("anneal", "sample"):
        smc.sro(lat, 3, occ, st["counts"], st["alpha"])
        out.update(counts=st["counts"], alpha=st["alpha"])
    if kind in ("stream", "sample"):
        smc.energy_grad(lat, model, occ, st["grad"])
        out["grad"] = st["grad"]
    smc.sweep(lat, model, occ, seed, s0, n, st["kT"], e_acc=e_acc, n_acc=n_acc)
    if kind == "job":
        smc.energy(lat, model, occ, e)
        smc.sro(lat, c["shells"], occ, st["counts"], st["alpha"])
        out.update(e=e, counts=st["counts"], alpha=st["alpha"])
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: the occupancy read once and written once (and read only, where
    nothing is swept), gradients written.  Operations: per trial the terms of
    the energy difference (two per neighbour of a and of b and shell) and one
    exponential's worth of arithmetic; network cases: the dense products of
    each distinct feature vector that the pass has to evaluate, never more
    than there are evaluations (40 per trial of unlike species) nor than there
    are feature vectors."""
    c = case
    n, sw = _sites(c), c.get("sweeps", 0)
    z = Z_FCC if c["kind"].startswith("fcc") else Z_BCC
    shells = c.get("shells", 3)
    flops = n * sw * (4.0 * sum(z[:shells]) + 10)
    vectors = c["S"] * float(np.prod([_compositions(m, c["S"]) for m in Z_BCC]))
    unlike = 1.0 - 1.0 / c["S"]
    byt = (2.0 if sw else 1.0) * n
    fwd, grad = 2 * (20 * 64 + 64 * 64 + 64), 29696
    if c["kind"] in ("mlp", "sample"):
        flops += fwd * min(n + n * sw * 40 * unlike, vectors)
    if c["kind"] == "mlpnet":
        flops += 2 * (20 * 96 + 2 * 96 * 96 + 96) * min(n + n * sw * 40 * unlike, vectors)
    if c["kind"] in ("sample", "fit"):
        flops += grad * min(n, vectors)
        byt += 4 * 5569
    return {"bytes": byt, "flops": flops}


def _compositions(m, S):
    """Ways to fill m neighbour sites with S species."""
    r = 1
    for i in range(S - 1):
        r = r * (m + i + 1) // (i + 1)
    return r


# ---------------------------------------------------------------------------
# 64-bit values of what is measured on the configuration a pass starts from.
# (The swept configuration follows from a chain of random decisions and is
# whole numbers; it has no value here.)
# ---------------------------------------------------------------------------
def _bcc_vectors(m, sub):
    """Shell m's (target sublattice, cell shift) from a site of sublattice sub."""
    if m == 0:
        o = (0, 1) if sub else (-1, 0)
        return [(1 - sub, v) for v in itertools.product(o, repeat=3)]
    want = 1 if m == 1 else 2
    return [(sub, v) for v in itertools.product((-1, 0, 1), repeat=3) if sum(map(abs, v)) == want]


_FCC_OFF = ((0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))


def _fcc_vectors(m, sub):
    out = []
    for v in itertools.product(range(-2, 3), repeat=3):
        if sum(x * x for x in v) == 2 * (m + 1) and sum(v) % 2 == 0:
            at = [o + x for o, x in zip(_FCC_OFF[sub], v)]
            out.append((_FCC_OFF.index(tuple(x % 2 for x in at)), tuple(x // 2 for x in at)))
    return out


def _neighbour(occ4, target, v):
    return torch.roll(occ4[target], shifts=(-v[2], -v[1], -v[0]), dims=(0, 1, 2))


def _pair_counts(occ4, S, shells, fcc):
    """Ordered pair counts [shells][S][S]."""
    out = torch.zeros((shells, S, S), dtype=torch.int64, device=occ4.device)
    for m in range(shells):
        for sub in range(occ4.shape[0]):
            for t, v in (_fcc_vectors if fcc else _bcc_vectors)(m, sub):
                o = _neighbour(occ4, t, v)
                for p in range(S):
                    mine = occ4[sub] == p
                    for q in range(S):
                        out[m, p, q] += (mine & (o == q)).sum()
    return out


def _alpha(cnt, n_p, z):
    n = float(n_p.sum())
    f = n_p.double() / n
    out = torch.empty(cnt.shape, dtype=torch.float64, device=cnt.device)
    for m in range(cnt.shape[0]):
        d = n * z[m] * f[:, None] * f[None, :]
        out[m] = torch.where(d > 0, 1.0 - cnt[m].double() / d, torch.full_like(d, float("nan")))
    return out


def _same_squares(occ4, S, shells, fcc):
    """Sum over sites of species p of their squared same-species count in shell m."""
    out = torch.zeros((shells, S), dtype=torch.float64, device=occ4.device)
    for m in range(shells):
        for sub in range(occ4.shape[0]):
            k = torch.zeros_like(occ4[sub], dtype=torch.int16)
            for t, v in (_fcc_vectors if fcc else _bcc_vectors)(m, sub):
                k += (_neighbour(occ4, t, v) == occ4[sub]).to(torch.int16)
            for p in range(S):
                out[m, p] += (k[occ4[sub] == p].double() ** 2).sum()
    return out


def _distinct_features(occ4, S):
    """The distinct MLP feature vectors [n, 20] (FP64) and how many sites have each."""
    keys = []
    for sub in range(2):
        key = occ4[sub].to(torch.int64)
        for m in range(3):
            part = torch.zeros_like(key)
            for t, v in _bcc_vectors(m, sub):
                part += torch.ones_like(key) << (4 * _neighbour(occ4, t, v).to(torch.int64))
            keep = (1 << 16) - 1  # species 0-3; the fifth count is what is left
            key = (key << 16) | (part & keep)
        keys.append(key.reshape(-1))
    u, cnt = torch.unique(torch.cat(keys), return_counts=True)
    x = torch.zeros((u.numel(), 20), dtype=torch.float64, device=u.device)
    for m in range(3):
        f = u >> (16 * (2 - m))
        left = torch.full_like(u, Z_BCC[m])
        for q in range(4):
            n = (f >> (4 * q)) & 15
            x[:, 5 + 5 * m + q] = n.double()
            left -= n
        x[:, 5 + 5 * m + 4] = left.double()
    x.scatter_(1, (u >> 48)[:, None], 1.0)
    return x, cnt.double()


def _mlp_exact(mlp, x, cnt, with_grad):
    w = {k: torch.tensor(inputs.bf16_bits_to_f32(mlp[k]).astype(np.float64), device=x.device) for k in ("w1", "w2", "w3")}
    w1, w2, w3 = w["w1"].reshape(64, 20), w["w2"].reshape(64, 64), w["w3"]
    b1, b2 = (torch.tensor(np.asarray(mlp[k], dtype=np.float64), device=x.device) for k in ("b1", "b2"))
    b3 = float(mlp["b3"])
    e, g = 0.0, [torch.zeros(s, dtype=torch.float64, device=x.device) for s in ((64, 20), 64, (64, 64), 64, 64, 1)]
    for i in range(0, x.shape[0], 1 << 20):
        xi, ci = x[i:i + (1 << 20)], cnt[i:i + (1 << 20)]
        z1 = xi @ w1.T + b1
        s1 = torch.sigmoid(z1)
        h1 = z1 * s1
        z2 = h1 @ w2.T + b2
        s2 = torch.sigmoid(z2)
        h2 = z2 * s2
        e += float((ci * (h2 @ w3 + b3)).sum())
        if with_grad:
            d2 = ci[:, None] * w3 * s2 * (1 + z2 * (1 - s2))
            d1 = (d2 @ w2) * s1 * (1 + z1 * (1 - s1))
            for k, v in enumerate((d1.T @ xi, d1.sum(0), d2.T @ h1, d2.sum(0), h2.T @ ci, ci.sum().reshape(1))):
                g[k] += v
    return e, torch.cat([v.reshape(-1) for v in g])


def _net_exact(net, x, cnt):
    w = [torch.tensor(inputs.bf16_bits_to_f32(net["w%d" % k]).astype(np.float64), device=x.device) for k in range(4)]
    b = [torch.tensor(np.asarray(net["b%d" % k], dtype=np.float64), device=x.device) for k in range(3)]
    e = 0.0
    for i in range(0, x.shape[0], 1 << 20):
        h = x[i:i + (1 << 20)]
        for k, n_in in enumerate((20, 96, 96)):
            h = torch.relu(h @ w[k].reshape(96, n_in).T + b[k])
        e += float((cnt[i:i + (1 << 20)] * (h @ w[3] + float(net["b3"]))).sum())
    return e


def exact(case, seed):
    c = dict(case)
    kind, S = c["kind"], c["S"]
    if kind in ("ladder", "job"):
        return None
    p = _parameters(c, seed)
    fcc = kind.startswith("fcc")
    occ = _occupancy(_sites(c), _fractions(c, seed), seed)
    occ4 = occ.reshape(4 if fcc else 2, c["nz"], c["ny"], c["nx"])
    z = Z_FCC if fcc else Z_BCC
    out = {}
    nsh = 3 if kind in ("anneal", "sample") else c.get("shells", 0)
    cnt = _pair_counts(occ4, S, nsh, fcc)
    if kind in ("small", "anneal", "fcc"):
        v = torch.tensor(np.asarray(p["v"], dtype=np.float64), device="cuda")
        unit = 1e-4 if fcc and c["integer"] else 1.0  # smc_fcc_energy gives eV, smc_energy the model's integer units
        out["e"] = (0.5 * unit * (v * cnt[:c["shells"]].double()).sum()).reshape(1)
    if kind in ("anneal", "sample"):
        out["alpha"] = _alpha(cnt, torch.bincount(occ.to(torch.int64), minlength=S), z)
    if kind in ("qsro", "fcc_qsro"):
        v, w = (torch.tensor(np.asarray(p[k], dtype=np.float64), device="cuda") for k in ("v", "w"))
        zz = torch.tensor(z[:nsh], dtype=torch.float64, device="cuda")
        e = (v * cnt.double() / zz[:, None, None]).sum() + (w * _same_squares(occ4, S, nsh, fcc) / zz[:, None] ** 2).sum()
        out["e"] = (e + occ.numel() * p["c"]).reshape(1)
    if kind in ("mlp", "mlpnet", "sample", "fit"):
        x, many = _distinct_features(occ4, S)
        if kind == "mlpnet":
            out["e"] = torch.tensor([_net_exact(p["net"], x, many)], dtype=torch.float64)
        else:
            e, g = _mlp_exact(p["mlp"], x, many, kind != "mlp")
            if kind == "mlp":
                out["e"] = torch.tensor([e], dtype=torch.float64)
    if kind in ("stream", "sample", "fit"):
        up = torch.triu_indices(S, S, device="cuda")
        pair = []
        for m in range(c["shells"]):
            d = cnt[m].double() - 0.5 * torch.diag(torch.diag(cnt[m].double()))
            pair.append(d[up[0], up[1]])
        pair = torch.cat(pair)
        out["grad"] = pair if kind == "stream" else torch.cat([pair, g])
    if kind == "fit":
        v = torch.tensor(np.asarray(p["v"], dtype=np.float64), device="cuda")
        out["e"] = (0.5 * (v * cnt.double()).sum() + e).reshape(())
    return out
