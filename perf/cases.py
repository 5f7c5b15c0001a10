"""What this library is asked to do, as cases that can be timed and checked.

A case is one call sequence of a user's program through the public entry points: forces of a given
configuration, a stretch of molecular dynamics (NVE, Nose-Hoover, stochastic bath; one system, a
batch of replicas, two dimensions; both precisions), the analysis calls, and the allocation-free
force call. Sizes are those of the repository's workloads (N = 1000, 32 000, 10^6, 8*10^6, the
512-replica mix, the 8 x 1000 cooling ladder, the planar model) and odd ones between them.

Configurations are Kob-Andersen liquids made here from the seed with plain tensor operations: a
small periodic box is melted from a jittered lattice, repeated to the size wanted, shaken a little,
thinned to the exact particle number, and given fresh Maxwell-Boltzmann velocities.

The mixed-precision path computes forces, velocities and pair energies in FP32, so what it returns
is taken in float32 here; the FP64 path's results are taken in float64. Positions are returned
unwrapped (x + L * image counter).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2001_07089_gb300 import kamd
from paper_2001_07089_gb300 import workloads as wl

DEV = "cuda" if torch.cuda.is_available() else "cpu"
DT = wl.DT
SIZES_MIX = "250,500,1000,2000,4000,8000"


def listed():
    return [
        # one energy/force evaluation of a configuration that an outer program proposes (a minimiser, a
        # Monte Carlo move, a calculator interface): the smallest call there is
        dict(name="forces_fp64_1000", kind="forces", precision="fp64", n=1000, T=1.0, **tuned("default")),
        # the same of a larger, odd-sized system in mixed precision
        dict(name="forces_mixed_100003", kind="forces", precision="mixed", n=100003, T=0.8, **tuned("default")),
        # forces inside a program that may not allocate (under stream capture, in a real-time loop)
        dict(name="noalloc_fp64_20011", kind="noalloc", precision="fp64", n=20011, T=1.0),
        # the paper's own run: N = 1000, NVE in double precision, thermodynamic record every 10 steps
        dict(name="nve_fp64_1000", kind="md", precision="fp64", n=1000, T=2.0, bath="nve", steps=100, log_every=10,
             **tuned("fp64_small")),
        # the double-precision arm of the N = 32 000 benchmark
        dict(name="nve_fp64_32000", kind="md", precision="fp64", n=32000, T=0.8, bath="nve", steps=40, log_every=10,
             **tuned("fp64")),
        # the N = 32 000 benchmark end to end: state from host memory, 100 NVE steps, log and state back
        dict(name="host_mixed_32000", kind="host", precision="mixed", n=32000, T=0.8, bath="nve", steps=100,
             log_every=10, **tuned("mid")),
        # the 10^6-particle thermostatted run
        dict(name="nvt_mixed_1000000", kind="md", precision="mixed", n=1000000, T=0.5, bath="nh", steps=50,
             log_every=10, **tuned("large")),
        # the largest system: NVE after the quench
        dict(name="nve_mixed_8000000", kind="md", precision="mixed", n=8000000, T=0.45, bath="nve", steps=20,
             log_every=10, **tuned("large")),
        # 512 independent replicas of uneven size, each with its own thermostat, in one launch
        dict(name="ensemble_512", kind="batch", precision="mixed", nrep=512, sizes=SIZES_MIX, mix=4, bath="nh",
             T_lo=0.45, T_hi=2.0, steps=50, log_every=10, **tuned("large")),
        # one rung of the cooling run sequence: 8 replicas, stochastic bath, then NVE
        dict(name="ladder_8x1000", kind="ladder", precision="mixed", nrep=8, sizes="1000", mix=6, T_lo=1.0, T_hi=1.0,
             steps=50, redraw=10, log_every=10, **tuned("small")),
        # partial g(r) to 4 sigma and the per-type MSD of a configuration on the way
        dict(name="analysis_mixed_1000000", kind="analysis", precision="mixed", n=1000000, T=0.5, dr=0.01, nbins=400,
             **tuned("large")),
        # the two-dimensional problem of the paper, thermostatted
        dict(name="plane_mixed_1000", kind="md", precision="mixed", n=1000, T=0.5, bath="nh_exact", steps=50,
             log_every=10, ndim=2, **tuned("small")),
    ]


# Launch configurations (threads_per_atom, block_size, skin, skin_outer): the library's default, and
# the ones that its autotuner settles on for the repository's workloads
TUNED = {
    "default": (4, 256, 0.3, 0.7),
    "small": (8, 512, 0.3, 1.0),
    "mid": (4, 512, 0.3, 1.4),
    "large": (1, 512, 0.4, 0.4),
    "fp64_small": (8, 256, 0.3, 1.2),
    "fp64": (1, 512, 0.3, 1.2),
}


def tuned(which):
    return dict(zip(("lanes", "block", "skin", "skin_outer"), TUNED[which]))


def draw(rng):
    """One more case: any of the kinds above at another size, temperature, bath and precision."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def fit(n, precision):
        if rng.random() < 0.25:
            return tuned("default")
        if precision == "fp64":
            return tuned("fp64_small" if n < 8000 else "fp64")
        return tuned("small" if n < 12000 else "mid" if n < 60000 else "large")

    kind = rng.choice(["forces", "noalloc", "md", "md", "md", "host", "batch", "ladder", "analysis", "plane"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    T = round(rng.uniform(0.45, 2.0), 3)
    steps = rng.randrange(20, 51)
    if kind == "forces":
        n = size(300, 300000 if precision == "mixed" else 60000)
        return dict(kind=kind, precision=precision, n=n, T=T, **fit(n, precision))
    if kind == "noalloc":
        return dict(kind=kind, precision="fp64", n=size(300, 131072), T=T)
    if kind == "md":
        n = size(300, 3000000 if precision == "mixed" else 50000)
        return dict(kind=kind, precision=precision, n=n, T=T, bath=rng.choice(["nve", "nve", "nh", "nh_exact"]),
                    steps=steps, log_every=10, **fit(n, precision))
    if kind == "plane":
        n = size(300, 30000)
        return dict(kind="md", precision=precision, n=n, T=round(rng.uniform(0.4, 1.0), 3),
                    bath=rng.choice(["nve", "nh"]), steps=steps, log_every=10, ndim=2, **fit(n, precision))
    if kind == "host":
        n = size(1000, 200000)
        return dict(kind=kind, precision="mixed", n=n, T=T, bath=rng.choice(["nve", "nh"]), steps=steps, log_every=10,
                    **fit(n, "mixed"))
    if kind == "batch":
        nrep = size(4, 512)
        return dict(kind=kind, precision="mixed", nrep=nrep, sizes=SIZES_MIX, mix=rng.randrange(1000),
                    bath=rng.choice(["nh", "nve"]), T_lo=0.45, T_hi=2.0, steps=steps, log_every=10,
                    **fit(2600 * nrep, "mixed"))
    if kind == "ladder":
        nrep, n = rng.randrange(2, 17), size(300, 3000)
        return dict(kind=kind, precision="mixed", nrep=nrep, sizes=str(n), mix=rng.randrange(1000), T_lo=T, T_hi=T,
                    steps=steps, redraw=rng.choice([5, 10, 25]), log_every=10, **fit(nrep * n, "mixed"))
    n = size(1000, 1000000 if precision == "mixed" else 100000)
    rmax = min(4.0, 0.49 * wl.box_length(n))
    nbins = rng.randrange(100, 401)
    return dict(kind="analysis", precision=precision, n=n, T=T, dr=rmax / nbins, nbins=nbins, **fit(n, precision))


# ------------------------------------------------------------------ inputs

def _melt(n, ndim, types, L, T, gen):
    """Positions (n, 3) of a small liquid: jittered lattice, all-pairs dynamics with the velocities
    scaled to T = 2 while it melts and then to T."""
    m = 1
    while m ** ndim < n:
        m += 1
    site = torch.arange(n, device=DEV, dtype=torch.int64) * (m ** ndim) // n
    k = torch.stack([site % m, (site // m) % m, site // (m * m)], 1).to(torch.float32)
    x = (k + 0.5) * (L / m) + 0.05 * (2.0 * torch.rand(n, 3, generator=gen, device=DEV) - 1.0)
    v = torch.randn(n, 3, generator=gen, device=DEV) * math.sqrt(2.0)
    if ndim == 2:
        x[:, 2] = 0.5 * L
        v[:, 2] = 0.0
    t = torch.from_numpy(types.astype(np.int64)).to(DEV)
    tab = [torch.tensor(a, dtype=torch.float32, device=DEV)[t][:, t] for a in (wl.KA_EPS, wl.KA_SIG ** 2, wl.KA_RC ** 2)]
    own = torch.eye(n, device=DEV) * 1e9

    def force(x):
        d = x[:, None, :] - x[None, :, :]
        d = d - L * torch.round(d / L)
        ir2 = 1.0 / ((d * d).sum(-1) + own)
        s6 = (tab[1] * ir2) ** 3
        w = torch.where(ir2 * tab[2] > 1.0, 48.0 * tab[0] * s6 * (s6 - 0.5) * ir2, 0.0)
        return (w[:, :, None] * d).sum(1)

    f = force(x)
    for step in range(240):
        if step % 5 == 0:
            v = v - v.mean(0)
            v = v * torch.sqrt((2.0 if step < 120 else T) * ndim * n / (v * v).sum())
        x = x + v * DT + f * (0.5 * DT * DT)
        fn = force(x)
        v = v + (f + fn) * (0.5 * DT)
        f = fn
    return x.to(torch.float64) % L


def _liquid(n, ndim, T, T_melt, seed, gen, bases):
    """(pos, vel, types, L) of n particles; `bases` keeps the small boxes already melted."""
    rho, frac_b = (wl.DENSITY, 0.2) if ndim == 3 else (wl.DENSITY_2D, wl.FRAC_B_2D)
    k = 1
    while k ** ndim * 1200 < n:
        k += 1
    nb = -(-n // k ** ndim)
    Lb = (nb / rho) ** (1.0 / ndim)
    if nb not in bases:
        tb = wl.ka_types(nb, seed, frac_b)
        bases[nb] = (_melt(nb, ndim, tb, Lb, T_melt, gen), tb)
    xb, tb = bases[nb]
    g = torch.arange(k, device=DEV, dtype=torch.float64)
    cell = torch.cartesian_prod(g, g, g if ndim == 3 else torch.zeros(1, device=DEV, dtype=torch.float64))
    L = k * Lb
    x = (cell[:, None, :] * Lb + xb[None]).reshape(-1, 3)
    x = x + 0.01 * torch.randn(x.shape, generator=gen, device=DEV, dtype=torch.float64)
    x = (x + L * torch.rand(3, generator=gen, device=DEV, dtype=torch.float64)) % L
    types = np.tile(tb, k ** ndim)
    if x.shape[0] > n:
        keep = torch.randperm(x.shape[0], generator=gen, device=DEV)[:n].sort().values
        x, types = x[keep], types[keep.cpu().numpy()]
    v = torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)
    if ndim == 2:
        x[:, 2] = 0.5 * L
        v[:, 2] = 0.0
    v = v - v.mean(0)
    v = v * torch.sqrt(T * ndim * n / (v * v).sum())
    return x.contiguous(), v.contiguous(), np.ascontiguousarray(types), L


def _inputs(case, seed):
    """Positions, velocities, types, and per replica: particle number, box edge, temperature."""
    gen = torch.Generator(device=DEV).manual_seed(1000003 * (seed % 1000000) + 17)
    ndim = case.get("ndim", 3)
    if "nrep" in case:
        spec = wl.ensemble(case["nrep"], case["mix"], [int(s) for s in case["sizes"].split(",")], case["T_lo"], case["T_hi"])
        n, T, melt_T = [int(k) for k in spec.n], [float(t) for t in spec.T], 1.0
    else:
        n, T, melt_T = [case["n"]], [case["T"]], case["T"]
    bases, parts = {}, []
    for r in range(len(n)):
        parts.append(_liquid(n[r], ndim, T[r], melt_T, seed, gen, bases))
    return dict(pos=torch.cat([p[0] for p in parts]), vel=torch.cat([p[1] for p in parts]),
                types=np.concatenate([p[2] for p in parts]), n=n, L=[p[3] for p in parts], T=np.array(T), ndim=ndim)


def _system(case, q):
    one = len(q["n"]) == 1
    s = kamd.System(q["n"][0] if one else q["n"], q["L"][0] if one else q["L"], q["types"], wl.KA_EPS, wl.KA_SIG,
                    wl.KA_RC, wl.KA_MASS, wl.SKIN, case["precision"], ndim=q["ndim"])
    s.set_tuning(case["lanes"], case["block"], case["skin"], case["skin_outer"])
    return s


def prepare(case, seed):
    q = _inputs(case, seed)
    kind, n = case["kind"], q["pos"].shape[0]
    st = dict(case=case, T=q["T"], seed=seed % 100000,
              real=torch.float32 if case["precision"] == "mixed" else torch.float64)
    if kind == "noalloc":
        st.update(pos=q["pos"], types=torch.from_numpy(q["types"]).to(DEV), n=n, L=q["L"][0],
                  f=torch.empty(n, 3, dtype=torch.float64, device=DEV),
                  pe=torch.empty(1, dtype=torch.float64, device=DEV), vir=torch.empty(1, dtype=torch.float64, device=DEV))
        return st
    s = _system(case, q)
    st["sys"] = s
    if kind == "host":
        def pinned(shape, dtype):
            return torch.empty(shape, dtype=dtype, pin_memory=DEV == "cuda")
        st["in"] = [pinned((n, 3), torch.float64).copy_(q[k].cpu()) for k in ("pos", "vel")]
        st["out"] = [pinned((n, 3), torch.float64), pinned((n, 3), torch.float64), pinned((n, 3), torch.int32)]
    else:
        st["in"] = [q["pos"], q["vel"]]
        st["out"] = [torch.empty(n, 3, dtype=torch.float64, device=DEV), torch.empty(n, 3, dtype=torch.float64, device=DEV),
                     torch.empty(n, 3, dtype=torch.int32, device=DEV)]
        s.set_state(q["pos"], q["vel"])
    st["L"] = torch.tensor(q["L"], dtype=torch.float64, device=st["out"][0].device)
    if len(q["n"]) > 1:  # each particle's box edge
        st["L"] = st["L"].repeat_interleave(torch.tensor(q["n"], device=st["L"].device))[:, None]
    if kind == "analysis":  # a little way from the reference positions, as between two measurements
        s.step_nve(DT, 5)
    return st


# ------------------------------------------------------------------ passes

def _thermo(log, real):
    real = np.float32 if real == torch.float32 else np.float64
    return {k: log[k] if k == "step" else log[k].astype(real) for k in log.dtype.names}


def _step(st, bath, steps, log_every):
    s, case = st["sys"], st["case"]
    if bath == "nve":
        return s.step_nve(DT, steps, log_every=log_every)
    if bath == "redraw":
        return s.step_nvt(DT, steps, st["T"], kind=kamd.MD_NVT_RESAMPLE, param=case["redraw"], seed=st["seed"],
                          log_every=log_every)
    kind = kamd.MD_NVT_NOSE_HOOVER if bath == "nh" else kamd.MD_NVT_NOSE_HOOVER_EXACT
    return s.step_nvt(DT, steps, st["T"], kind=kind, param=100 * DT, log_every=log_every)


def run(st):
    case, real = st["case"], st["real"]
    kind = case["kind"]
    if kind == "noalloc":
        kamd.md_forces_noalloc(st["n"], st["pos"], st["types"], 2, st["L"], wl.KA_EPS, wl.KA_SIG, wl.KA_RC, st["f"],
                               st["pe"], st["vir"])
        return {"f": st["f"], "pe": st["pe"], "virial": st["vir"]}
    s = st["sys"]
    if kind == "forces":
        s.set_state(st["in"][0])
        f = st["out"][0]
        pe, vir = np.zeros(s.nrep), np.zeros(s.nrep)
        kamd.md_forces(s.handle, f, pe, vir, on_device=1)
        if real == torch.float32:
            pe, vir = pe.astype(np.float32), vir.astype(np.float32)
        return {"f": f.to(real), "pe": pe, "virial": vir}
    if kind == "analysis":
        g = s.rdf(case["dr"], case["nbins"], reset=True)
        m = s.msd()
        return {"g": g.astype(np.float32), "msd": m.astype(np.float32)} if real == torch.float32 else {"g": g, "msd": m}
    pos, vel, img = st["out"]
    if kind == "host":
        kamd.md_set_state(s.handle, st["in"][0].numpy(), st["in"][1].numpy())
        log = _step(st, case["bath"], case["steps"], case["log_every"])
        kamd.md_get_state(s.handle, pos.numpy(), vel.numpy(), img.numpy(), 0)
    else:
        if kind == "ladder":
            half = case["steps"] // 2
            log = np.concatenate([_step(st, "redraw", half, case["log_every"]),
                                  _step(st, "nve", case["steps"] - half, case["log_every"])])
        else:
            log = _step(st, case["bath"], case["steps"], case["log_every"])
        s.get_state_device(pos, vel, img)
    out = _thermo(log, real)
    out["pos"] = torch.addcmul(pos, img.to(pos.dtype), st["L"]).to(real)
    out["vel"] = vel.to(real)
    return out


# ------------------------------------------------------------------ work

def _count(case):
    """(particles, interacting pairs per particle, replicas)."""
    if "nrep" in case:
        n = int(wl.ensemble(case["nrep"], case["mix"], [int(s) for s in case["sizes"].split(",")]).n.sum())
        nrep = case["nrep"]
    else:
        n, nrep = case["n"], 1
    if case.get("ndim", 3) == 2:
        x, vol = (1 - wl.FRAC_B_2D, wl.FRAC_B_2D), lambda r: math.pi * r * r * wl.DENSITY_2D
    else:
        x, vol = (0.8, 0.2), lambda r: 4.0 / 3.0 * math.pi * r ** 3 * wl.DENSITY
    half = 0.5 * sum(x[a] * x[b] * vol(float(wl.KA_RC[a, b])) for a in range(2) for b in range(2))
    return n, half, nrep


def work(case):
    """Each array in and out of the call once; every pair inside the cutoff once per force evaluation
    (26 operations with its energy), 30 operations per particle and step for the integration."""
    n, half, nrep = _count(case)
    if case["kind"] in ("forces", "noalloc"):
        return {"bytes": float(n * (24 + 1 + 24)), "flops": float(n * half * 26)}
    if case["kind"] == "analysis":
        pairs = n * 0.5 * 4.0 / 3.0 * math.pi * (case["dr"] * case["nbins"]) ** 3 * wl.DENSITY
        return {"bytes": float(n * (24 + 1 + 36 + 24) + 24 * case["nbins"]), "flops": float(pairs * 10 + n * 10)}
    steps = case["steps"]
    state_in = n * (24 + 24 + 1)
    state_out = n * (24 + 24 + 12)
    log = 64 * nrep * (steps // case["log_every"])
    return {"bytes": float(state_in + state_out + log), "flops": float(steps * n * (26 * half + 30))}


# ------------------------------------------------------------------ 64-bit results

EPS, SIG2, RC = (torch.tensor(a, dtype=torch.float64, device=DEV) for a in (wl.KA_EPS, wl.KA_SIG ** 2, wl.KA_RC))
SR6 = (SIG2 / (RC * RC)) ** 3
VSH = 4.0 * EPS * (SR6 * SR6 - SR6)
REACH = 0.5  # how far the pair lists below reach past the largest cutoff


def _close(x, L, reach, visit):
    """Calls visit(i, j, d) for the pairs of one box nearer than `reach`, each pair once, in blocks."""
    n = x.shape[0]
    nc = min(int(L / reach), 256)

    def pairs(i, j, keep):
        d = x[i] - x[j]
        d -= L * torch.round(d / L)
        keep &= (d * d).sum(-1) < reach * reach
        i, j = i.expand(keep.shape)[keep], j.expand(keep.shape)[keep]
        visit(i, j, d[keep])

    if nc < 4 or n <= 3000:
        rows = max(1, (1 << 24) // n)
        every = torch.arange(n, device=x.device)
        for a in range(0, n, rows):
            i = every[a:a + rows, None]
            pairs(i, every[None, :], every[None, :] > i)
        return
    c = torch.clamp((x * (nc / L)).to(torch.int64), 0, nc - 1)
    key = (c[:, 2] * nc + c[:, 1]) * nc + c[:, 0]
    order = torch.argsort(key, stable=True)
    count = torch.bincount(key, minlength=nc ** 3)
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    table = torch.full((nc ** 3, cap), -1, dtype=torch.int64, device=x.device)
    ks = key[order]
    table[ks, torch.arange(n, device=x.device) - start[ks]] = order
    ids = torch.arange(nc ** 3, device=x.device)
    ids = ids[count > 0]
    cx, cy, cz = ids % nc, (ids // nc) % nc, ids // (nc * nc)
    block = max(1, (1 << 24) // (cap * cap))
    for oz in (-1, 0, 1):
        for oy in (-1, 0, 1):
            for ox in (-1, 0, 1):
                if (oz, oy, ox) < (0, 0, 0):
                    continue
                nb = (((cz + oz) % nc) * nc + (cy + oy) % nc) * nc + (cx + ox) % nc
                for a in range(0, ids.numel(), block):
                    i, j = table[ids[a:a + block]][:, :, None], table[nb[a:a + block]][:, None, :]
                    keep = (i >= 0) & (j >= 0)
                    keep = keep & (j > i) if (oz, oy, ox) == (0, 0, 0) else keep.clone()
                    pairs(i.clamp(min=0), j.clamp(min=0), keep)


class _Plain:
    """The dynamics of the paper in 64-bit tensor operations, all replicas together."""

    def __init__(self, q):
        self.ndim, self.nL = q["ndim"], q["L"]
        self.n = torch.tensor(q["n"], device=DEV)
        self.rep = torch.repeat_interleave(torch.arange(len(q["n"]), device=DEV), self.n)
        self.L = torch.tensor(q["L"], dtype=torch.float64, device=DEV)
        self.t = torch.from_numpy(q["types"].astype(np.int64)).to(DEV)
        self.x, self.v = q["pos"].clone(), q["vel"].clone()
        self.T = torch.tensor(q["T"], dtype=torch.float64, device=DEV)
        self.X = self.ndim * self.n.to(torch.float64)
        self.step, self.xi, self.lns = 0, torch.zeros_like(self.T), torch.zeros_like(self.T)
        self.listed_at = None

    def lists(self):
        self.ij, o = [], 0
        for r, n in enumerate(self.n.tolist()):
            L, found = self.nL[r], []
            _close(self.x[o:o + n] % L, L, min(float(RC.max()) + REACH, 0.5 * L), lambda i, j, d: found.append(torch.stack([i, j])))
            self.ij += [f.to(torch.int32) + o for f in found]
            o += n
        if len(self.ij) > 64:
            self.ij = list(torch.cat(self.ij, 1).split(1 << 25, 1))
        self.listed_at = self.x.clone()

    def forces(self):
        # a box under twice the reach lists its nearest images out to L/2 only: list those afresh each time
        small = min(self.nL) < 2 * (float(RC.max()) + REACH)
        if self.listed_at is None or small or float(((self.x - self.listed_at) ** 2).sum(-1).max()) > (0.5 * REACH) ** 2:
            self.lists()
        f = torch.zeros_like(self.x)
        nrep = self.n.numel()
        self.pe, self.vir = (torch.zeros(nrep, dtype=torch.float64, device=DEV) for _ in range(2))
        for ij in self.ij:
            i, j = ij[0].to(torch.int64), ij[1].to(torch.int64)
            r = self.rep[i]
            L = self.L[r][:, None]
            d = self.x[i] - self.x[j]
            d -= L * torch.round(d / L)
            r2 = (d * d).sum(-1)
            ti, tj = self.t[i], self.t[j]
            near = r2 < (RC * RC)[ti, tj]
            s6 = (SIG2[ti, tj] / r2) ** 3
            w = torch.where(near, 48.0 * EPS[ti, tj] * s6 * (s6 - 0.5), 0.0)
            self.vir.index_add_(0, r, w)
            self.pe.index_add_(0, r, torch.where(near, 4.0 * EPS[ti, tj] * s6 * (s6 - 1.0) - VSH[ti, tj], 0.0))
            d *= (w / r2)[:, None]
            f.index_add_(0, i, d)
            f.index_add_(0, j, d, alpha=-1.0)
        return f

    def per_rep(self, v):
        return torch.zeros(self.n.numel(), dtype=torch.float64, device=DEV).index_add_(0, self.rep, v)

    def kinetic(self):
        return 0.5 * self.per_rep((self.v * self.v).sum(-1))

    def redraw(self, seed, number):
        first = torch.cumsum(self.n, 0) - self.n
        p = (torch.arange(self.x.shape[0], device=DEV) - first[self.rep]).cpu().numpy()
        g = torch.from_numpy(_normals(seed, number, p)).to(DEV)
        if self.ndim == 2:
            g[:, 2] = 0.0
        v = g * torch.sqrt(self.T[self.rep])[:, None]
        nn = self.n.to(torch.float64)
        v = v - torch.stack([self.per_rep(v[:, c]) / nn for c in range(3)], 1)[self.rep]
        self.v = v * torch.sqrt(self.X * self.T / self.per_rep((v * v).sum(-1)))[self.rep][:, None]

    def go(self, bath, steps, log_every, redraw=0, seed=0):
        h, rows = 0.5 * DT, []
        nh = bath in ("nh", "nh_exact")
        Q = self.X * self.T * (100 * DT) ** 2
        f = self.forces()
        g = (2.0 * self.kinetic() - self.X * self.T) / Q if nh else None
        for k in range(1, steps + 1):
            self.step += 1
            if nh:
                xa = self.xi + DT * g
                lns = self.lns + self.xi * DT + 0.5 * g * DT * DT
                xi_p, xa_p = self.xi[self.rep][:, None], xa[self.rep][:, None]
                self.x = self.x + self.v * DT + (f - xi_p * self.v) * (h * DT)
            else:
                self.x = self.x + self.v * DT + f * (h * DT)
            fn = self.forces()
            if bath == "nh":
                self.v = self.v + h * ((f + fn) - (xi_p + xa_p) * self.v) * (1.0 - h * xa_p)
            elif bath == "nh_exact":
                self.v = (self.v + h * (f - xi_p * self.v + fn)) / (1.0 + h * xa_p)
            else:
                self.v = self.v + h * (f + fn)
            f = fn
            if nh:
                gn = (2.0 * self.kinetic() - self.X * self.T) / Q
                self.xi, self.lns, g = self.xi + h * (g + gn), lns, gn
            if bath == "redraw" and self.step % redraw == 0:
                self.redraw(seed, self.step // redraw)
            if k % log_every == 0:
                ke, n = self.kinetic(), self.n.to(torch.float64)
                H = ke + self.pe + (0.5 * Q * self.xi ** 2 + self.X * self.T * self.lns if nh else 0.0)
                rows.append(dict(step=torch.full_like(self.n, self.step), T=2.0 * ke / self.X, pe_per_n=self.pe / n,
                                 ke_per_n=ke / n, etot_per_n=(ke + self.pe) / n, virial=self.vir, h_nh=H,
                                 xi=self.xi if nh else torch.zeros_like(n)))
        return rows


def _normals(seed, number, p):
    """Three standard normals per particle index: Philox4x32-10 (Salmon et al., SC'11) and Box-Muller."""
    m32 = np.uint64(0xFFFFFFFF)
    z = []
    for blk in range(2):
        c = [p.astype(np.uint64), np.full(p.shape, number & 0xFFFFFFFF, np.uint64),
             np.full(p.shape, (2 << 16) | blk, np.uint64), np.full(p.shape, number >> 32, np.uint64)]
        k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
        for _ in range(10):
            a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
            c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & m32, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & m32]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        u = [(((c[q] << np.uint64(21)) ^ (c[q + 1] >> np.uint64(11))).astype(np.float64) + 0.5) / 2.0 ** 53 for q in (0, 2)]
        rad = np.sqrt(-2.0 * np.log(u[0]))
        z += [rad * np.cos(2.0 * np.pi * u[1]), rad * np.sin(2.0 * np.pi * u[1])]
    return np.stack(z[:3], 1)


def _histogram(x, t, L, dr, nbins):
    """Partial g(r) of one configuration: AA, BB, AB."""
    h = torch.zeros(3, nbins, dtype=torch.float64, device=DEV)

    def add(i, j, d):
        k = (torch.sqrt((d * d).sum(-1)) / dr).to(torch.int64)
        a, b = t[i], t[j]
        which = torch.where(a != b, 2, a)
        ok = k < nbins
        h.view(-1).add_(torch.bincount((which * nbins + k)[ok], minlength=3 * nbins).to(torch.float64))

    _close(x % L, L, dr * nbins * (1.0 + 1e-12), add)
    nb = int(t.sum())
    na = t.numel() - nb
    k = torch.arange(nbins, dtype=torch.float64, device=DEV)
    shell = 4.0 / 3.0 * math.pi * ((k + 1) ** 3 - k ** 3) * dr ** 3
    norm = torch.tensor([2.0 / (na * (na - 1)), 2.0 / (nb * (nb - 1)), 1.0 / (na * nb)], dtype=torch.float64, device=DEV)
    return h / shell * L ** 3 * norm[:, None]


def exact(case, seed):
    q = _inputs(case, seed)
    p = _Plain(q)
    kind = case["kind"]
    if kind in ("forces", "noalloc"):
        f = p.forces()
        return {"f": f, "pe": p.pe, "virial": p.vir}
    if kind == "analysis":
        x0 = p.x
        p.go("nve", 5, 100)
        d2 = ((p.x - x0) ** 2).sum(-1)
        msd = torch.stack([d2[p.t == a].mean() for a in range(2)])
        return {"g": _histogram(p.x, p.t, q["L"][0], case["dr"], case["nbins"]), "msd": msd}
    if kind == "ladder":
        half = case["steps"] // 2
        rows = p.go("redraw", half, case["log_every"], case["redraw"], seed % 100000)
        rows += p.go("nve", case["steps"] - half, case["log_every"])
    else:
        rows = p.go(case["bath"], case["steps"], case["log_every"])
    out = {k: torch.stack([r[k] for r in rows]) for k in rows[0]}
    out["pos"], out["vel"] = p.x, p.v
    return out
