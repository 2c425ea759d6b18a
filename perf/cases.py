"""Performance cases of the XY engines: what is timed, over which ranges.

Each case is one pass through the Python front ends (``lattice.Lattice``,
``lattice.Batch``, ``lattice.Quad``, ``hmc.HMC``, ``autograd.chain_averages``),
as a simulation program calls them.  ``listed`` names the cases, ``draw`` gives
more of the same ranges, ``prepare`` builds what a program holds before the
pass, ``run`` is the pass with whole outputs (angles, per-sweep or
per-trajectory observables, gradients), ``work`` its unavoidable bytes and
floating-point operations, and ``exact`` the same outputs from plain FP64 torch
where such a value exists.
"""
import math

import numpy as np
import torch

from paper_0811_2111_gb300.autograd import chain_averages
from paper_0811_2111_gb300.hmc import HMC
from paper_0811_2111_gb300.lattice import Batch, Lattice, Quad
from paper_0811_2111_gb300.workloads import (BATCH_BETA_GRID, BATCH_LS, batch_layout,
                                             hmc_step_for, random_angles)

TWO_PI = 2.0 * math.pi
# A chain of Metropolis decisions has an FP64 counterpart only while no accept
# test falls within FP32 rounding of its threshold (about 1e-7 per update):
# from the first such test on the two chains are different samples.
EXACT_UPDATES = 200_000


def listed():
    return [
        # the smallest call: a few sweeps of a small lattice, then its observables, as
        # an interactive program or a measuring loop makes them (latency and launches)
        dict(name="lattice_L64", kind="lattice", L=64, beta=1.0, sweeps=10, sincos="accurate",
             reduce="exact"),
        # the repository's small validation workload: one long chain of L = 32
        dict(name="lattice_L32_chain", kind="lattice", L=32, beta=1.0, sweeps=1000,
             sincos="accurate", reduce="exact"),
        # a mid-size lattice of the paper's Table 1: less than a wave of work per sweep
        dict(name="lattice_L512", kind="lattice", L=512, beta=1.0, sweeps=200, sincos="accurate",
             reduce="exact"),
        # a side that is no multiple of any tile (finite-size studies take any even side)
        dict(name="lattice_L1000", kind="lattice", L=1000, beta=1.12, sweeps=100,
             sincos="accurate", reduce="exact"),
        # the headline throughput lattice
        dict(name="lattice_L4096", kind="lattice", L=4096, beta=1.12, sweeps=100,
             sincos="accurate", reduce="exact"),
        # the largest production side (1 GiB of angles), SFU sincos
        dict(name="lattice_L16384_fast", kind="lattice", L=16384, beta=1.12, sweeps=10,
             sincos="fast", reduce="exact"),
        # checkpoint -> sweeps -> checkpoint, with CUDA's sincosf and compensated sums
        # (the precision study's other options)
        dict(name="resume_L2048_libm", kind="resume", L=2048, beta=1.12, sweeps=100,
             sincos="libm", reduce="compensated"),
        # the 256-lattice replica-exchange workload: 8 ladders of uneven sides
        dict(name="batch_exchange", kind="batch", ladders=8, per_ladder=32, rounds=20,
             sweeps_per_round=10),
        # d<O>/dbeta: 41 chains of L = 256, forward and backward
        dict(name="chains_autograd", kind="chains", L=256, chains=41, therm=500, meas=2000),
        # Hybrid Monte Carlo at the throughput side: unit trajectories, then the state
        dict(name="hmc_L4096", kind="hmc", L=4096, beta=1.12, traj=8, sincos="accurate"),
        # a small HMC chain of the reference step size (eps = 0.1, ten steps)
        dict(name="hmc_L64", kind="hmc", L=64, beta=1.0, traj=50, sincos="accurate"),
        # four replicas per site at four temperatures (the RGBA packing)
        dict(name="quad_L1024", kind="quad", L=1024, sweeps=100, sincos="accurate"),
    ]


def _side(rng, lo, hi, multiple=2):
    """An even side, log-uniform in [lo, hi]; one time in three a multiple of 128."""
    L = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    m = 128 if hi >= 256 and L >= 128 and rng.random() < 1 / 3 else multiple
    return max(lo, min(hi, L // m * m))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "resume", "batch", "chains", "hmc", "hmc",
                       "quad"])
    beta = round(rng.uniform(0.8, 1.4), 4)
    sincos = rng.choice(["accurate", "accurate", "fast", "libm"])
    if kind in ("lattice", "resume"):
        L = _side(rng, 16, 8192 if kind == "lattice" else 2048)
        return dict(kind=kind, L=L, beta=beta, sweeps=_log_int(rng, 5, min(1000, 4.0e8 / L ** 2)),
                    sincos=sincos, reduce=rng.choice(["exact", "exact", "compensated"]))
    if kind == "batch":
        return dict(kind=kind, ladders=rng.randint(1, 8), per_ladder=rng.randint(2, 32),
                    rounds=rng.randint(1, 20), sweeps_per_round=rng.randint(5, 20))
    if kind == "chains":
        L = _side(rng, 16, 256)
        chains = rng.randint(2, 41)
        return dict(kind=kind, L=L, chains=chains, therm=100 * rng.randint(1, 3),
                    meas=100 * rng.randint(2, 8))
    if kind == "hmc":
        L = _side(rng, 16, 4096)
        return dict(kind=kind, L=L, beta=beta,
                    traj=_log_int(rng, 1, min(50, max(1.0, 4.0e7 / L ** 2))), sincos=sincos)
    L = _side(rng, 16, 2048)
    return dict(kind=kind, L=L, sweeps=_log_int(rng, 5, min(300, 1.0e8 / L ** 2)), sincos=sincos)


def _quad_betas():
    return [1.0, 1.06, 1.12, 1.18]


def _batch_lists(case):
    """(Ls, betas, ladders): the 256-lattice layout, or the same scheme with fewer ladders
    (largest sides first) and lattices per ladder."""
    if case["ladders"] == len(BATCH_LS) and case["per_ladder"] == 32:
        return batch_layout()
    Ls, betas, ladders = [], [], []
    for i, L in enumerate(sorted(BATCH_LS, reverse=True)[:case["ladders"]]):
        for j in range(case["per_ladder"]):
            Ls.append(L)
            betas.append(BATCH_BETA_GRID[(i % 2) + 2 * j])
            ladders.append(i)
    return Ls, betas, ladders


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case, seed=seed)
    if kind in ("lattice", "resume"):
        s["engine"] = Lattice(case["L"], case["beta"], seed, sincos=case["sincos"],
                              reduce=case["reduce"])
        s["engine"].reserve(case["sweeps"])
        if kind == "resume":
            s["checkpoint"] = random_angles(case["L"], seed)
    elif kind == "batch":
        Ls, betas, ladders = _batch_lists(case)
        s["engine"] = Batch(Ls, betas, seed, ladders=ladders,
                            sweeps_per_round=case["sweeps_per_round"])
        s["engine"].reserve(100 * case["rounds"])
        s["done"] = 0
    elif kind == "chains":
        s["beta"] = torch.linspace(0.9, 1.3, case["chains"], dtype=torch.float64, device="cuda",
                                   requires_grad=True)
    elif kind == "hmc":
        eps, n_md = hmc_step_for(case["L"])
        s["engine"] = HMC(case["L"], case["beta"], seed, eps, n_md, sincos=case["sincos"])
        s["done"] = 0
    else:
        s["engine"] = Quad(case["L"], _quad_betas(), seed, sincos=case["sincos"])
        s["done"] = 0
    return s


def _plain(obs):
    """Observables with the accept counts as signed integers."""
    return {k: v.astype(np.int64) if v.dtype.kind == "u" else v for k, v in obs.items()}


def run(s):
    kind = s["kind"]
    if kind == "lattice":
        # an independent chain: start from the seed, sweep, measure every sweep
        lat = s["engine"]
        lat.reset(s["seed"])
        lat.sweep(s["sweeps"])
        return {"observables": _plain(lat.observables()), "angles": lat.angles}
    if kind == "resume":
        lat = s["engine"]
        lat.set_state(s["checkpoint"], 0)
        lat.sweep(s["sweeps"])
        obs = _plain(lat.observables())
        return {"observables": obs, "angles": lat.state()[0]}
    if kind == "batch":
        # the chains go on from pass to pass, as a run's rounds do; after a block of rounds
        # a program looks at the exchange and at each ladder's last lattice: the last
        # round's series and the configuration
        b = s["engine"]
        n = s["sweeps_per_round"]
        b.run(s["rounds"])
        s["done"] += s["rounds"] * n
        slots, accepted, attempted = b.exchange_stats()
        last = [(i + 1) * s["per_ladder"] - 1 for i in range(s["ladders"])]
        obs = [_plain(b.observables(i, s["done"] - n, n)) for i in last]
        return {"observables": {k: np.stack([o[k] for o in obs]) for k in obs[0]},
                "betas": b.betas(), "slots": slots, "swaps": accepted.astype(np.int64),
                "tries": attempted.astype(np.int64), "angles": [b.state(i) for i in last]}
    if kind == "chains":
        beta = s["beta"]
        beta.grad = None
        e, u = chain_averages(beta, s["L"], s["seed"], s["therm"], s["meas"])
        (e.sum() + u.sum()).backward()
        return {"e": e.detach(), "upsilon": u.detach(), "grad": beta.grad}
    if kind == "hmc":
        h = s["engine"]
        first = s["done"]
        h.run(s["traj"])
        s["done"] = first + s["traj"]
        obs = _plain(h.observables(first, s["traj"]))
        angles, momenta, _ = h.state()
        return {"observables": obs, "angles": angles, "momenta": momenta}
    q = s["engine"]
    first = s["done"]
    q.sweep(s["sweeps"])
    s["done"] = first + s["sweeps"]
    return {"observables": [_plain(q.observables(r, first, s["sweeps"])) for r in range(4)],
            "angles": [q.state(r)[0] for r in range(4)]}


# Floating-point operations of one site update: proposal and wrap 5, the proposal's
# unit vector 26, neighbour sums 6, energy change and Boltzmann test 16, half of a
# black site's five sums 10; of one leap-frog site-step: unit vector 26, neighbour
# sums 6, force 4, kick, drift and wrap 10.
UPDATE_FLOPS = 63.0
STEP_FLOPS = 46.0


def work(case):
    kind = case["kind"]
    if kind in ("lattice", "resume"):
        n = case["L"] ** 2
        return {"bytes": (8.0 if kind == "resume" else 4.0) * n + 64.0 * case["sweeps"],
                "flops": UPDATE_FLOPS * n * case["sweeps"]}
    if kind == "batch":
        Ls, _, _ = _batch_lists(case)
        n = float(sum(L * L for L in Ls))
        sweeps = case["rounds"] * case["sweeps_per_round"]
        return {"bytes": 8.0 * n + 64.0 * len(Ls) * sweeps, "flops": UPDATE_FLOPS * n * sweeps}
    if kind == "chains":
        n = float(case["chains"] * case["L"] ** 2)
        sweeps = case["therm"] + case["meas"]
        return {"bytes": 4.0 * n + 64.0 * case["chains"] * sweeps,
                "flops": UPDATE_FLOPS * n * sweeps}
    n = float(case["L"] ** 2)
    if kind == "hmc":
        n_md = hmc_step_for(case["L"])[1]
        return {"bytes": 12.0 * n + 128.0 * case["traj"],
                "flops": STEP_FLOPS * n * n_md * case["traj"]}
    return {"bytes": 32.0 * n + 256.0 * case["sweeps"],
            "flops": 4.0 * UPDATE_FLOPS * n * case["sweeps"]}


# ---- the same method in FP64 torch --------------------------------------------------------

def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words (int64 tensors holding 32-bit values) of the counters."""
    mask = 0xFFFFFFFF
    k0, k1 = seed & mask, (seed >> 32) & mask
    x = [c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.full_like(c0, c3)]
    for _ in range(10):
        a, b = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
        x = [((b >> 32) & mask) ^ x[1] ^ k0, b & mask, ((a >> 32) & mask) ^ x[3] ^ k1, a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return x


def _u24(w):
    return (w >> 8).double() / 16777216.0


def _hot(L, seed):
    site = torch.arange(L * L, dtype=torch.int64, device="cuda")
    return (TWO_PI * _u24(_philox(site, 0, 0, 0, seed)[0])).view(L, L)


def _neighbours(v):
    return v.roll(1, 1) + v.roll(-1, 1) + v.roll(1, 0) + v.roll(-1, 0)


def _bond_sums(th):
    """[C, Ix, Iy, Mx, My] of a state (one row), every bond counted once."""
    dx, dy = th - th.roll(-1, 1), th - th.roll(-1, 0)
    return torch.stack([dx.cos().sum() + dy.cos().sum(), dx.sin().sum(), dy.sin().sum(),
                        th.cos().sum(), th.sin().sum()])


def _observables(rows, accepted, beta, N):
    C, Ix, Iy, Mx, My = torch.stack(rows).cpu().numpy().T
    return {"C": C, "Ix": Ix, "Iy": Iy, "Mx": Mx, "My": My, "e": -C / N,
            "abs_m": np.sqrt(Mx ** 2 + My ** 2) / N,
            "upsilon": (C - beta * (Ix ** 2 + Iy ** 2)) / (2 * N),
            "beta": np.full(len(C), beta), "accepted": np.array(accepted, np.int64)}


def _exact_lattice(case, seed):
    L, beta = case["L"], case["beta"]
    if L * L * case["sweeps"] > EXACT_UPDATES:
        return None
    if case["kind"] == "resume":
        th = torch.from_numpy(random_angles(L, seed)).to("cuda", torch.float64)
    else:
        th = _hot(L, seed)
    y, x = torch.meshgrid(torch.arange(L, device="cuda"), torch.arange(L, device="cuda"),
                          indexing="ij")
    counter = (y * L + x - (x & 2)).reshape(-1)
    rows, accepted = [], []
    for sweep in range(case["sweeps"]):
        w = [v.view(L, L) for v in _philox(counter, sweep, 0, 1, seed)]
        u0 = _u24(torch.where((x & 2) != 0, w[2], w[0]))
        u1 = _u24(torch.where((x & 2) != 0, w[3], w[1]))
        n_acc = 0
        for colour in (0, 1):
            tp = th + math.pi * (2.0 * u0 - 1.0)
            tp = torch.where(tp < 0, tp + TWO_PI, torch.where(tp >= TWO_PI, tp - TWO_PI, tp))
            sc, ss = _neighbours(th.cos()), _neighbours(th.sin())
            gain = (tp.cos() - th.cos()) * sc + (tp.sin() - th.sin()) * ss
            take = (((x + y) & 1) == colour) & (u1 < torch.exp(beta * gain))
            th = torch.where(take, tp, th)
            n_acc += int(take.sum())
        rows.append(_bond_sums(th))
        accepted.append(n_acc)
    obs = _observables(rows, accepted, beta, L * L)
    if case["kind"] == "resume":
        return {"observables": obs, "angles": th.cpu().numpy()}
    # the working buffer's order: [colour][y][x >> 1]
    split = torch.stack([torch.stack([th[r, (c + r) % 2::2] for r in range(L)]) for c in (0, 1)])
    return {"observables": obs, "angles": split.reshape(-1)}


def _exact_hmc(case, seed):
    L, beta = case["L"], case["beta"]
    eps, n_md = hmc_step_for(L)
    if L * L * n_md * case["traj"] > 1.2e10:
        return None
    site = torch.arange(L * L, dtype=torch.int64, device="cuda")
    zero = torch.zeros(1, dtype=torch.int64, device="cuda")

    def force(th):
        c, s = th.cos(), th.sin()
        return beta * (c * _neighbours(s) - s * _neighbours(c))

    th, rows, accepted, dHs, p = _hot(L, seed), [], [], [], None
    for traj in range(case["traj"]):
        w = _philox(site, traj, 0, 3, seed)
        u1 = ((w[0] >> 8).double() + 1.0) / 16777216.0
        p = ((-2.0 * u1.log()).sqrt() * (TWO_PI * _u24(w[1])).cos()).view(L, L)
        del w, u1
        old = th
        start = _bond_sums(old)
        h0 = 0.5 * p.square().sum() - beta * start[0]
        p = p + 0.5 * eps * force(th)
        for step in range(n_md):
            th = torch.remainder(th + eps * p, TWO_PI)
            p = p + (eps if step + 1 < n_md else 0.5 * eps) * force(th)
        end = _bond_sums(th)
        dH = float(0.5 * p.square().sum() - beta * end[0] - h0)
        u = float(_u24(_philox(zero, traj, 0, 4, seed)[0]))
        take = u < math.exp(min(0.0, -dH))
        if not take:
            th = old
        rows.append(end if take else start)
        accepted.append(int(take))
        dHs.append(dH)
    obs = _observables(rows, accepted, beta, L * L)
    obs["dH"] = np.array(dHs)
    return {"observables": obs, "angles": th.cpu().numpy(), "momenta": p.cpu().numpy()}


def exact(case, seed):
    if case["kind"] in ("lattice", "resume"):
        return _exact_lattice(case, seed)
    if case["kind"] == "hmc":
        return _exact_hmc(case, seed)
    # batches, four-replica lattices and differentiated chains are long Metropolis chains
    # (see EXACT_UPDATES)
    return None
