"""Performance cases of the library: what a user has it do, through its public entry points.

A case is a dict of plain values.  Three kinds:

``lattice``   one lattice on the GPU (``Simulation`` with caller-owned torch buffers): a pass is one
              ``step(steps)`` call, with the sampled observables of that call where ``sample_every`` > 0,
              and its outputs are the stored populations (the handle's own device buffer) and the
              observables.
``ensemble``  many independent lattices of one type (``Ensemble``): a pass is one ``step(steps)`` call and
              the read-out of every member.
``served``    a batch of requests to the continuous-batching server (``Server``): a pass submits them and
              drains the server; the outputs are the requests' final populations in host memory.

``exact`` restates the method (Wagner & Strand, arXiv:1606.07801) in 64-bit torch without the library:
Philox4x32-10 words, Box-Muller or flat variates, the Gram-Schmidt moment basis, the moment-space
collision and the periodic pull.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1606_07801_gb300 as lb
from paper_1606_07801_gb300 import synth

LATTICE = {"d1q3": lb.D1Q3, "d2q9": lb.D2Q9, "d3q19": lb.D3Q19, "d2q5": lb.D2Q5}
PRECISION = {"f32": lb.F32, "f64": lb.F64, "f16": lb.F32_F16, "bf16": lb.F32_BF16}
NOISE = {"local": lb.NOISE_LOCAL, "global": lb.NOISE_GLOBAL, "off": lb.NOISE_OFF}
LAW = {"gauss": lb.GAUSSIAN, "flat": lb.UNIFORM}
BYTES = {"f32": 4, "f64": 8, "f16": 2, "bf16": 2}
TORCH = {"f32": torch.float32, "f64": torch.float64, "f16": torch.float16, "bf16": torch.bfloat16}
Q_OF = {"d1q3": 3, "d2q5": 5, "d2q9": 9, "d3q19": 19}
D_OF = {"d1q3": 1, "d2q5": 2, "d2q9": 2, "d3q19": 3}
# structure-factor modes a sampled run takes (at most four)
MODES = {"d1q3": [(1, 0, 0), (2, 0, 0)], "d2q5": [(1, 0, 0), (2, 0, 0), (0, 1, 0)],
         "d2q9": [(1, 0, 0), (2, 0, 0), (0, 1, 0)], "d3q19": [(1, 0, 0), (2, 0, 0), (0, 1, 0), (1, 1, 1)]}


def _lattice(name, lattice, dims, steps, *, precision="f32", noise="local", law="gauss", tau=0.8, rho=100.0,
             sample_every=0, mrt=False, theta=0.0):
    d = list(dims) + [1] * (3 - len(dims))
    case = {"kind": "lattice", "lattice": lattice, "nx": d[0], "ny": d[1], "nz": d[2], "steps": steps,
            "precision": precision, "noise": noise, "law": law, "tau": tau, "rho": rho, "sample_every": sample_every,
            "mrt": mrt, "theta": theta}
    return {"name": name} | case if name else case


def listed():
    return [
        # the FP64 line of the paper's 1-D check: 256 sites, a thousand steps a call; latency is everything
        _lattice("line_d1q3_f64", "d1q3", (256,), 1000, precision="f64", tau=1.0, rho=10.0),
        # the paper's own lattice at the size of its time-correlator experiment, flat noise, the moments
        # relaxed with their own times: a small lattice on the moment-space kernel
        _lattice("paper_d2q5_mrt", "d2q5", (81, 81), 200, law="flat", tau=1.0, rho=120.0, mrt=True, theta=1.0 / 3.0),
        # a small FP32 plane stepped a hundred times a call, as in a parameter study
        _lattice("small_d2q9_f32", "d2q9", (64, 48), 100, rho=100.0),
        # single-lattice throughput in two dimensions: the plane of the benchmark
        _lattice("plane_d2q9_f32", "d2q9", (2048, 2048), 20, rho=100.0),
        # odd and ragged sides, the other noise mode and the paper's flat law
        _lattice("odd_d2q9_f32", "d2q9", (1023, 771), 20, noise="global", law="flat", tau=1.1, rho=20.0),
        # FP64 reference runs with sampled equilibrium statistics
        _lattice("plane_d2q9_f64", "d2q9", (512, 384), 10, precision="f64", tau=0.9, rho=50.0, sample_every=10),
        # the plane of the benchmark with its observables sampled every ten steps
        _lattice("sampled_d2q9_f32", "d2q9", (2048, 2048), 20, rho=100.0, sample_every=10),
        # single-lattice throughput in three dimensions, FP32 storage, and 16-bit storage
        _lattice("cube_d3q19_f32", "d3q19", (256, 256, 256), 6, tau=1.0, rho=50.0),
        _lattice("cube_d3q19_f16", "d3q19", (256, 256, 256), 6, precision="f16", tau=1.0, rho=50.0),
        # the moments of D3Q19 relaxed with their own times
        _lattice("cube_d3q19_mrt", "d3q19", (128, 120, 96), 10, tau=1.0, rho=60.0, mrt=True),
        # an ensemble of uneven planes run for the two thousand steps of its production runs and read out
        {"name": "ensemble_d2q9_f32", "kind": "ensemble", "lattice": "d2q9", "precision": "f32", "members": 60,
         "side_lo": 96, "side_hi": 512, "steps": 2000},
        # a mixed stream served to completion
        {"name": "served_mixed_f32", "kind": "served", "precision": "f32", "requests": 24, "steps_lo": 100,
         "steps_hi": 2000, "d1_hi": 65536, "d2_hi": 1024, "d3_hi": 128},
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Site updates of one drawn pass at most, per lattice (FP64 sites cost more)
UPDATES = {"d1q3": 6e7, "d2q5": 6e7, "d2q9": 6e7, "d3q19": 6e7}


def draw(rng):
    u = rng.random()
    if u < 0.08:
        return {"kind": "ensemble", "lattice": rng.choice(["d2q9", "d2q9", "d3q19"]),
                "precision": rng.choice(["f32", "f32", "f16"]), "members": _logu(rng, 4, 60),
                "side_lo": rng.choice([20, 32, 50]), "side_hi": _logu(rng, 60, 100), "steps": _logu(rng, 100, 1000)}
    if u < 0.14:
        return {"kind": "served", "precision": "f32", "requests": _logu(rng, 4, 24), "steps_lo": 50,
                "steps_hi": _logu(rng, 100, 1000), "d1_hi": _logu(rng, 1000, 65536), "d2_hi": _logu(rng, 64, 512),
                "d3_hi": _logu(rng, 40, 64)}
    lattice = rng.choice(["d1q3", "d2q5", "d2q9", "d2q9", "d2q9", "d3q19", "d3q19"])
    mrt = lattice == "d2q5" or rng.random() < 0.12
    precision = rng.choice(["f32", "f32", "f64"]) if mrt else rng.choice(["f32", "f32", "f32", "f16", "bf16", "f64"])
    hi = {"d1q3": 1 << 22, "d2q5": 1 << 22, "d2q9": 1 << 22, "d3q19": 1 << 23}[lattice]
    n = _logu(rng, 256, hi // (8 if precision == "f64" else 1))
    D = D_OF[lattice]
    if D == 1:
        dims = (n,)
    else:
        side = n ** (1.0 / D)
        dims = [max(3, int(round(side * math.exp(rng.uniform(-0.6, 0.6))))) for _ in range(D - 1)]
        dims = tuple(dims + [max(3, n // max(1, int(np.prod(dims))))])
        if rng.random() < 0.5:  # a side of whole vectors, as users mostly choose
            dims = (max(4, dims[0] // 8 * 8),) + dims[1:]
    sites = int(np.prod(dims))
    most = UPDATES[lattice] / (16 if precision == "f64" else 1)
    steps = max(2, min(_logu(rng, 3, 1000), int(most / sites)))
    every = rng.choice([0, 0, 0, 5, 10]) if steps >= 5 else 0
    return _lattice(None, lattice, dims, steps, precision=precision, noise=rng.choice(["local", "local", "global", "off"]),
                    law=rng.choice(["gauss", "gauss", "flat"]), tau=round(rng.uniform(0.6, 1.5), 3),
                    rho=round(rng.uniform(20.0, 200.0), 2), sample_every=every, mrt=mrt,
                    theta=round(rng.uniform(0.1, 0.45), 3) if lattice == "d2q5" else 0.0)


# ---- inputs --------------------------------------------------------------------------------------------------

def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _taus(case):
    """tau^a of the moments a = 0 .. Q-1: spread around tau where the case relaxes them apart."""
    q = Q_OF[case["lattice"]]
    if not case["mrt"]:
        return [case["tau"]] * q
    return [case["tau"]] + [round(case["tau"] * (0.75 + 0.5 * ((7 * a) % q) / q), 4) for a in range(1, q)]


def _weights(case):
    if case["lattice"] == "d1q3":
        return [2 / 3, 1 / 6, 1 / 6]
    if case["lattice"] == "d2q9":
        return [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    if case["lattice"] == "d3q19":
        return [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    th = case["theta"] or 1 / 3
    return [1 - 2 * th] + [th / 2] * 4


def _state(case, seed):
    """The stored state [Q, N] a run starts from: populations in thermal equilibrium around a density with one
    long wave of 5% (their variance is their mean, as the method's is), as deviations from w_i rho_mean for the
    16-bit formats."""
    q, (nx, ny, nz) = Q_OF[case["lattice"]], _dims(case)
    n, rho, w = nx * ny * nz, case["rho"], _weights(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)
    wave = (0.05 * rho) * torch.sin(2 * math.pi * torch.arange(nx, device="cuda", dtype=torch.float32) / nx)
    wave = wave.repeat(ny * nz)
    compute = torch.float64 if case["precision"] == "f64" else torch.float32
    out = torch.empty((q, n), device="cuda", dtype=TORCH[case["precision"]])
    for i in range(q):
        z = torch.empty(n, device="cuda", dtype=compute).normal_(0.0, math.sqrt(w[i] * rho), generator=g)
        z += w[i] * wave
        if case["precision"] in ("f32", "f64"):
            z += w[i] * rho
        out[i] = z.to(out.dtype)
    return out


def _modes(case):
    return MODES[case["lattice"]] if case["sample_every"] else []


def _ensemble_specs(case, seed):
    """The members: their sizes belong to the case, their densities, relaxation times and noise seeds to the seed."""
    ndim = D_OF[case["lattice"]]
    sizes = synth.ensemble(case["members"], case["side_lo"], case["side_hi"], seed=12345, ndim=ndim)
    drawn = synth.ensemble(case["members"], case["side_lo"], case["side_hi"], seed=int(seed) + 1, ndim=ndim)
    return [d | {"dims": s["dims"]} for s, d in zip(sizes, drawn)]


def _served_specs(case, seed):
    """The requests, in the mix and ranges of the benchmark's trace: sizes and step counts belong to the case."""
    def trace(k):
        return synth.served_trace(case["requests"], seed=k, d1_range=(256, case["d1_hi"]), d2_side=(32, case["d2_hi"]),
                                  d3_side=(32, case["d3_hi"]), steps_range=(case["steps_lo"], case["steps_hi"]))[1]
    return [d | {k: s[k] for k in ("lattice", "dims", "steps")} for s, d in zip(trace(777), trace(int(seed) + 1))]


def prepare(case, seed):
    if case["kind"] == "lattice":
        sim = lb.Simulation(LATTICE[case["lattice"]], _dims(case), case["tau"], case["rho"], int(seed) + 1,
                            precision=PRECISION[case["precision"]], noise_mode=NOISE[case["noise"]],
                            noise_dist=LAW[case["law"]], init=lb.INIT_NONE, modes=_modes(case), torch_buffers=True,
                            theta=case["theta"], tau_moments=_taus(case) if case["mrt"] else None,
                            sample_every=case["sample_every"])
        state = {"case": case, "sim": sim}
        _current(state).copy_(_state(case, seed))
        return state
    if case["kind"] == "ensemble":
        ens = lb.Ensemble(LATTICE[case["lattice"]], _ensemble_specs(case, seed), precision=PRECISION[case["precision"]])
        # the decomposition the tuner picks for such an ensemble: parameter-bank tiles of eight passes
        ens.plan(2, 8, 0, lb.WALK_PARAM)
        return {"case": case, "ens": ens}
    specs = _served_specs(case, seed)
    server = lb.Server(precision=PRECISION[case["precision"]], hbm_budget=8 << 30, passes=4, solo_sites=0,
                       walk=lb.WALK_PARAM, policy=lb.POLICY_SHORTEST, max_active_sites=20_000_000)
    outs = [torch.empty((lb.Q_OF[s["lattice"]], int(np.prod(s["dims"]))), dtype=torch.float32, pin_memory=True)
            for s in specs]
    return {"case": case, "server": server, "specs": specs, "outs": outs}


def _current(state):
    """The handle's current device buffer as [Q, N]."""
    sim = state["sim"]
    ptr = sim.state_device()[0]
    buf = sim.buffers[0] if sim.buffers[0].data_ptr() == ptr else sim.buffers[1]
    return buf.view(sim.Q, sim.N)


# ---- one pass ------------------------------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "lattice":
        sim = state["sim"]
        if not case["sample_every"]:
            sim.step(case["steps"])
            return {"state": _current(state)}
        sim.reset_obs()
        sim.step(case["steps"])
        ob = sim.observables()
        # FP32-arithmetic lattices take these sums in FP32 over tiles of sites: they are good to FP32
        kind = np.float64 if case["precision"] == "f64" else np.float32
        return {"state": _current(state), "t": ob["t"], "n_samples": ob["n_samples"],
                "rho": np.array([ob["sum_rho"]], dtype=kind), "rho2": np.array([ob["sum_rho2"]], dtype=kind),
                "f": ob["sum_f"].astype(kind), "ff": ob["sum_ff"].astype(kind), "sk": ob["sum_sk"].astype(kind)}
    if case["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        return [ens.get_f(m).astype(np.float32) for m in range(case["members"])]
    server = state["server"]
    for s, out in zip(state["specs"], state["outs"]):
        server.submit(s["lattice"], s["dims"], s["tau"], s["rho_mean"], s["seed"], s["steps"],
                      lattice_id=s["lattice_id"], result=lb.RESULT_F, out=out.numpy())
    server.drain()
    return state["outs"]


# ---- what a pass cannot do without ---------------------------------------------------------------------------

def _site_ops(lattice, noise, mrt):
    """Arithmetic of one site update: density, relaxation (2 per population, or both transforms), and for the
    noise 15 integer operations a Philox word, 10 for each variate, and the back-transform."""
    q = Q_OF[lattice]
    transform = {"d1q3": 6, "d2q5": 30, "d2q9": 48, "d3q19": 232}[lattice]
    ops = 5 * q + (2 * transform + 3 * q if mrt else 0)
    if noise != "off":
        ops += 25 * (q - 1) + (0 if mrt else transform)
    return ops


def work(case):
    if case["kind"] == "lattice":
        q, n = Q_OF[case["lattice"]], case["nx"] * case["ny"] * case["nz"]
        ops = float(case["steps"]) * n * _site_ops(case["lattice"], case["noise"], case["mrt"])
        if case["sample_every"]:
            samples = (case["steps"] + case["sample_every"] - 1) // case["sample_every"]
            ops += float(samples) * n * (q * (q + 1) + 2 * q + 8 * len(_modes(case)))
        return {"bytes": 2.0 * q * n * BYTES[case["precision"]], "flops": ops}
    if case["kind"] == "ensemble":
        sites = float(sum(int(np.prod(s["dims"])) for s in _ensemble_specs(case, 0)))
        q = Q_OF[case["lattice"]]
        return {"bytes": sites * q * (2 * BYTES[case["precision"]] + 8),
                "flops": sites * case["steps"] * _site_ops(case["lattice"], "local", False)}
    names = {v: k for k, v in LATTICE.items()}
    total, ops = 0.0, 0.0
    for s in _served_specs(case, 0):
        n, name = float(np.prod(s["dims"])), names[s["lattice"]]
        total += n * Q_OF[name] * 4
        ops += n * s["steps"] * _site_ops(name, "local", False)
    return {"bytes": total, "flops": ops}


# ---- the same in 64 bits, without the library ------------------------------------------------------------------

_V = {
    "d1q3": [(0, 0, 0), (1, 0, 0), (-1, 0, 0)],
    "d2q5": [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)],
    "d2q9": [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
    "d3q19": [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)],
}


def _basis(case):
    """m[a][i]: weighted Gram-Schmidt over the lattice's list of monomials of the velocity."""
    name = case["lattice"]
    v, w = np.array(_V[name], dtype=float), np.array(_weights(case))
    x, y, z = v.T
    if name == "d1q3":
        seeds = [x ** 0, x, x * x]
    elif name == "d2q9":
        seeds = [x ** p * y ** r for p in range(3) for r in range(3)]
    elif name == "d2q5":
        seeds = [x ** 0, x, y, x * x - y * y, x * x + y * y]
    else:
        powers = [(p, r, s) for p in range(3) for r in range(3) for s in range(3) if (p > 0) + (r > 0) + (s > 0) <= 2]
        powers.sort(key=lambda e: (sum(e), -e[0], -e[1], -e[2]))
        seeds = [x ** p * y ** r * z ** s for p, r, s in powers]
    rows = []
    for u in seeds:
        u = u.copy()
        for b in rows:
            u = u - (u * w * b).sum() * b
        u = u / math.sqrt((u * w * u).sum())
        u[np.abs(u) < 1e-13] = 0.0
        rows.append(u)
    return np.array(rows)


def _philox(site, lid, t, j, seed):
    """The four words of call j at every site (Philox4x32-10), as int64 tensors of 32-bit values."""
    mask = 0xFFFFFFFF
    c = [site, torch.full_like(site, lid), torch.full_like(site, t & mask),
         torch.full_like(site, (((t >> 32) * 8) + j) & mask)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # the low 64 bits of the products
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _variates(site, count, t, seed, law):
    z = []
    for j in range((count + 3) // 4):
        u = [((r >> 8).double() + 0.5) * 2.0 ** -24 for r in _philox(site, 0, t, j, seed)]
        if law == "flat":
            z += [math.sqrt(3.0) * (2.0 * x - 1.0) for x in u]
        else:
            for a in (0, 2):
                rad, ang = torch.sqrt(-2.0 * torch.log(u[a])), 2.0 * math.pi * u[a + 1]
                z += [rad * torch.cos(ang), rad * torch.sin(ang)]
    return z[:count]


def exact(case, seed):
    if case["kind"] != "lattice":
        return None  # thousands of steps of dozens of lattices: minutes in 64 bits
    q, (nx, ny, nz) = Q_OF[case["lattice"]], _dims(case)
    n = nx * ny * nz
    if case["steps"] * max(n, 200_000) * q > 3.5e9:
        return None
    w, v, m, taus, rho_mean = _weights(case), _V[case["lattice"]], _basis(case), _taus(case), case["rho"]
    off = [w[i] * rho_mean if case["precision"] in ("f16", "bf16") else 0.0 for i in range(q)]
    g = _state(case, seed).double()
    for i in range(q):
        g[i] += off[i]
    site = torch.arange(n, device="cuda", dtype=torch.int64)
    every, samples = case["sample_every"], 0
    sums = [torch.zeros(1, device="cuda", dtype=torch.float64), torch.zeros(1, device="cuda", dtype=torch.float64),
            torch.zeros(q, device="cuda", dtype=torch.float64), torch.zeros(q, q, device="cuda", dtype=torch.float64)]
    sk = torch.zeros(len(_modes(case)), device="cuda", dtype=torch.float64)
    for t in range(case["steps"]):
        f = [torch.roll(g[i].view(nz, ny, nx), (v[i][2], v[i][1], v[i][0]), (0, 1, 2)).reshape(n) for i in range(q)]
        rho = f[0].clone()
        for i in range(1, q):
            rho += f[i]
        if every and t % every == 0:
            samples += 1
            sums[0] += rho.sum()
            sums[1] += (rho * rho).sum()
            for i in range(q):
                sums[2][i] += f[i].sum()
                for j in range(i, q):
                    s = torch.dot(f[i], f[j])
                    sums[3][i, j] += s
                    if i != j:
                        sums[3][j, i] += s
            for a, (kx, ky, kz) in enumerate(_modes(case)):
                ph = 2 * math.pi * ((kx * (site % nx) % nx).double() / nx + (ky * (site // nx % ny) % ny).double() / ny +
                                    (kz * (site // (nx * ny)) % nz).double() / nz)
                d = rho - rho_mean
                sk[a] += torch.dot(d, torch.cos(ph)) ** 2 + torch.dot(d, torch.sin(ph)) ** 2
        if case["noise"] != "off":
            z = _variates(site, q - 1, t, int(seed) + 1, case["law"])
            base = torch.sqrt(torch.clamp(rho, min=0.0)) if case["noise"] == "local" else math.sqrt(rho_mean)
        # moment by moment: relax, add the noise, and add its share to every population
        new = [w[i] * rho for i in range(q)]
        for a in range(1, q):
            M = torch.zeros_like(rho)
            for i in range(q):
                if m[a][i] != 0.0:
                    M += m[a][i] * f[i]
            M *= 1.0 - 1.0 / taus[a]
            if case["noise"] != "off":
                M += (math.sqrt(2.0 * taus[a] - 1.0) / taus[a]) * base * z[a - 1]
            for i in range(q):
                if m[a][i] != 0.0:
                    new[i] += (w[i] * m[a][i]) * M
        g = torch.stack(new)
    for i in range(q):
        g[i] -= off[i]
    out = {"state": g}
    if every:
        out |= {"t": None, "n_samples": None, "rho": sums[0], "rho2": sums[1], "f": sums[2], "ff": sums[3], "sk": sk}
    return out
