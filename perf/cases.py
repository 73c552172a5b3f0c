"""The performance cases: what users of the library run, through its public entry points.

A case names a kind of work, the instance family and its sizes, and the solve's
parameters in plain values. Instances and start states come from the seed.

Outputs are what the call returns. Whole solves under the paper's stopping rule,
and low-temperature schedules on low-precision tensor cores, amplify a last-bit
difference into other local minima, so ``exact`` has no 64-bit value for them
(their energies, spins and counts are compared with each other instead); it has
one for noisy mean-field annealing and for energies of given spins.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_1907_05124_gb300 import instances, mars

K_MAX, D_MIN = 1000, 1e-4


def listed():
    return [
        # The smallest whole solve: a toy lattice, as in a first try or a unit
        # test. Launches, host work and a lone replica's latency count.
        dict(name="ea2d_L12_R64", kind="solve", family="ea", dim=2, size=12, replicas=64,
             t_max=4.0, levels=4, sweeps=0, precision="fp32", method="mars"),
        # The 2-D +-J spin glass of the benchmark: 10^4 spins, 1024 replicas,
        # every replica's state on chip.
        dict(name="ea2d_L100_R1024", kind="solve", family="ea", dim=2, size=100, replicas=1024,
             t_max=4.0, levels=4, sweeps=0, precision="fp32", method="mars"),
        # A cubic lattice beyond shared memory: replicas resident in HBM, one
        # grid-wide launch per colour level.
        dict(name="ea3d_L64_R256", kind="solve", family="ea", dim=3, size=64, replicas=256,
             t_max=6.0, levels=6, sweeps=0, precision="fp32", method="mars"),
        # Max-cut shaped random graphs of mixed size and degree with a cubic
        # lattice, solved as one batch (uneven instances, uneven replicas).
        dict(name="batch_er_mix", kind="batch", jobs=6, size=2000, replicas=512),
        # The paper's smallest SK study: 64 spins, every pair coupled, FP32.
        dict(name="sk_pm1_64_fp32", kind="solve", family="sk_pm1", size=64, replicas=256,
             t_max=16.0, levels=16, sweeps=0, precision="fp32", method="mars"),
        # A mid-sized dense instance on the FP32 path, Gaussian couplings (the
        # exact FP64 energies of non-integer couplings are part of it).
        dict(name="sk_gauss_256_fp32", kind="solve", family="sk_gauss", size=256, replicas=512,
             t_max=2.0, levels=32, sweeps=0, precision="fp32", method="mars"),
        # Noisy mean-field annealing (synchronous sweeps) on a dense instance.
        dict(name="nmfa_gauss_1024", kind="solve", family="sk_gauss", size=1024, replicas=512,
             t_max=2.0, levels=32, sweeps=1, precision="fp32", method="nmfa"),
        # The time-to-target configuration: a whole BF16 tensor-core solve.
        dict(name="sk_gauss_1024_bf16", kind="solve", family="sk_gauss", size=1024, replicas=256,
             t_max=2.0, levels=64, sweeps=0, precision="bf16", method="mars"),
        # The benchmark's dense configuration (8192 spins, 4096 replicas) under
        # a fixed budget of sweeps per level, as a deadline-bound user runs it.
        dict(name="sk_gauss_8192_bf16", kind="solve", family="sk_gauss", size=8192, replicas=4096,
             t_max=2.0, levels=64, sweeps=2, precision="bf16", method="mars"),
        # +-1 couplings on E4M3 tensor cores, fixed budget, the serving mix's size.
        dict(name="sk_pm1_4096_fp8", kind="solve", family="sk_pm1", size=4096, replicas=1024,
             t_max=128.0, levels=64, sweeps=8, precision="fp8", method="mars"),
        # Energies of spin vectors found elsewhere (checking or ranking
        # another solver's samples).
        dict(name="energy_gauss_2048", kind="energy", family="sk_gauss", size=2048, count=512),
        # Serving: requests of the serving mix submitted together and polled
        # until every one is done.
        dict(name="serve_mix_16", kind="serve", requests=16, size=64, replicas=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ea2d", "ea2d", "ea3d", "ea3d_hbm", "er", "batch", "dense", "dense", "nmfa",
                       "nmfa_sparse", "bf16", "bf16_fixed", "fp8_fixed", "energy", "energy_sparse",
                       "serve"])
    mars_ = dict(kind="solve", sweeps=0, precision="fp32", method="mars")
    if kind == "ea2d":
        return dict(mars_, family="ea", dim=2, size=_log_int(rng, 8, 110), replicas=_log_int(rng, 16, 1024),
                    t_max=4.0, levels=4)
    if kind == "ea3d":
        return dict(mars_, family="ea", dim=3, size=_log_int(rng, 5, 32), replicas=_log_int(rng, 16, 512),
                    t_max=6.0, levels=6)
    if kind == "ea3d_hbm":
        return dict(mars_, family="ea", dim=3, size=rng.randint(39, 64), replicas=_log_int(rng, 16, 256),
                    t_max=6.0, levels=6)
    if kind == "er":
        n = _log_int(rng, 200, 20000)
        d = rng.choice([4, 6, 12, 24, 40]) if n < 6000 else rng.choice([4, 6])
        return dict(mars_, family="er", size=n, degree=d, weights=rng.choice(["one", "pm1"]),
                    replicas=_log_int(rng, 32, 512), t_max=2.0 * d ** 0.5 + 1.0, levels=round(2.0 * d ** 0.5 + 1.0))
    if kind == "batch":
        return dict(kind="batch", jobs=rng.randint(2, 6), size=_log_int(rng, 300, 2000),
                    replicas=_log_int(rng, 64, 512))
    if kind == "dense":
        n = _log_int(rng, 24, 320)
        fam = rng.choice(["sk_pm1", "sk_gauss"])
        return dict(mars_, family=fam, size=n, replicas=_log_int(rng, 16, 512),
                    t_max=round(2.0 * n ** 0.5, 3) if fam == "sk_pm1" else 2.0,
                    levels=max(4, round(2.0 * n ** 0.5)))
    if kind == "nmfa":
        return dict(mars_, family=rng.choice(["sk_gauss", "sk_uniform"]), size=_log_int(rng, 100, 2048),
                    replicas=_log_int(rng, 32, 512), t_max=2.0, levels=rng.choice([8, 16, 32]), sweeps=1,
                    method="nmfa")
    if kind == "nmfa_sparse":
        return dict(mars_, family="er", size=_log_int(rng, 500, 8000), degree=rng.choice([4, 6, 12]), weights="pm1",
                    replicas=_log_int(rng, 32, 512), t_max=2.0, levels=rng.choice([16, 32]), sweeps=1, method="nmfa")
    if kind == "bf16":
        n = rng.randint(256, 1024)
        return dict(mars_, family="sk_gauss", size=n, replicas=_log_int(rng, 64, 256), t_max=2.0,
                    levels=rng.choice([32, 64]), precision="bf16")
    if kind == "bf16_fixed":
        n = _log_int(rng, 512, 8192)
        return dict(mars_, family="sk_gauss", size=n, replicas=_log_int(rng, 64, 4096), t_max=2.0,
                    levels=rng.choice([16, 32, 64]), sweeps=rng.choice([1, 2]), precision="bf16")
    if kind == "fp8_fixed":
        n = _log_int(rng, 512, 8192)
        return dict(mars_, family="sk_pm1", size=n, replicas=_log_int(rng, 64, 4096),
                    t_max=round(2.0 * n ** 0.5, 3), levels=rng.choice([16, 32, 64]), sweeps=rng.choice([2, 4, 8]),
                    precision="fp8")
    if kind == "energy":
        return dict(kind="energy", family=rng.choice(["sk_gauss", "sk_pm1"]), size=_log_int(rng, 60, 4096),
                    count=_log_int(rng, 1, 1024))
    if kind == "energy_sparse":
        return dict(kind="energy", family="er", size=_log_int(rng, 200, 50000), degree=rng.choice([4, 6, 12, 40]),
                    weights="pm1", count=_log_int(rng, 1, 1024))
    return dict(kind="serve", requests=rng.randint(4, 24), size=rng.randint(24, 64), replicas=_log_int(rng, 64, 256))


class _State:
    """A context, its registered instances and the call's arguments."""

    def __init__(self):
        self.ctx = mars.Context(0)


def _dense(case, seed):
    """Dense couplings on the GPU: float32 Gaussian or uniform, int8 +-1."""
    n = case["size"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["family"] == "sk_gauss":
        u = torch.randn(n, n, generator=g, device="cuda") / n ** 0.5
    elif case["family"] == "sk_uniform":
        u = (2.0 * torch.rand(n, n, generator=g, device="cuda") - 1.0) * (3.0 / n) ** 0.5
    else:
        u = torch.where(torch.rand(n, n, generator=g, device="cuda") < 0.5, -1.0, 1.0)
    u = torch.triu(u, 1)
    u = u + u.T
    return u.to(torch.int8) if case["family"] == "sk_pm1" else u.contiguous()


def _sparse(case, seed):
    if case["family"] == "ea":
        return instances.ea_lattice(case["size"], case["dim"], seed)
    return instances.er_graph(case["size"], case["degree"], seed, case.get("weights", "pm1"))


def _spins(case, seed):
    g = np.random.default_rng(seed + 77)
    return np.where(g.random((case["count"], case["size"])) < 0.5, -1, 1).astype(np.int8)


def _start(case, seed):
    """Start states and temperatures of a caller that draws its own."""
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    m0 = 2.0 * torch.rand(case["replicas"], case["size"], generator=g, device="cuda") - 1.0
    t0 = case["t_max"] * torch.rand(case["replicas"], generator=g, device="cuda")
    return m0, t0


def prepare(case, seed):
    s = _State()
    s.kind, s.case, s.seed = case["kind"], case, seed
    if case["kind"] == "batch":
        rng = np.random.default_rng(seed)
        s.jobs = []
        for j in range(case["jobs"]):
            # sizes and degrees as in the benchmark's batch, the last a lattice
            n = max(64, int(case["size"] * (0.4, 1.0, 0.7, 1.0, 0.5)[j % 5]))
            d = (6, 40, 12, 6, 24)[j % 5]
            if j == case["jobs"] - 1:
                g, t_max = instances.ea_lattice(max(3, round(n ** (1 / 3))), 3, seed + j), 6.0
            else:
                g = instances.er_graph(n, d, seed + j, "one" if j % 2 else "pm1")
                t_max = d + 1.0 if j % 2 else 2.0 * d ** 0.5 + 1.0
            R = max(16, case["replicas"] >> (j % 3))
            s.jobs.append((s.ctx.add_csr(*g), R, 0.0, t_max, dict(c_step=1.0, seed=int(rng.integers(1 << 30)))))
        return s
    if case["kind"] == "serve":
        ctx = s.ctx
        L, R = case["size"], case["replicas"]
        # lattices, random graphs and small dense instances, as in the serving mix
        pool = [(ctx.add_csr(*instances.ea_lattice(L, 2, seed)), 4.0, 1.0, "fp32"),
                (ctx.add_csr(*instances.ea_lattice(max(4, L // 4), 3, seed + 1)), 6.0, 1.0, "fp32"),
                (ctx.add_csr(*instances.er_graph(16 * L, 12, seed + 2)), 8.0, 1.0, "fp32"),
                (ctx.add_dense(instances.sk_pm1(2 * L, seed + 3)), 2.0 * (2 * L) ** 0.5, 1.0, "fp32"),
                (ctx.add_csr(*instances.er_graph(64 * L, 4, seed + 4)), 5.0, 1.0, "fp32"),
                (ctx.add_dense(instances.sk_gauss(8 * L, seed + 5)), 2.0, 0.125, "bf16")]
        ctx.serve_limits(16)
        s.requests = [(pool[q % 6], max(16, R >> (q % 3)), seed * 100 + q) for q in range(case["requests"])]
        return s
    dense = case["family"].startswith("sk_")
    s.inst = s.ctx.add_dense(_dense(case, seed)) if dense else s.ctx.add_csr(*_sparse(case, seed))
    if case["kind"] == "energy":
        s.spins = _spins(case, seed)
        return s
    s.kw = dict(c_step=case["t_max"] / case["levels"], d_min=D_MIN, k_max=K_MAX, precision=case["precision"], seed=seed)
    if case["method"] == "nmfa":
        s.kw.update(method="nmfa", alpha=0.5, sigma=0.15, outputs=("energies", "m_final"), device_outputs=True)
        s.kw["m0"], s.kw["t0"] = _start(case, seed)
    elif case["sweeps"]:
        # a caller on the GPU: outputs stay there
        s.kw.update(fixed_sweeps=case["sweeps"], outputs=("energies", "m_final", "spins", "levels"),
                    device_outputs=True)
    else:
        s.kw.update(outputs=("energies", "m_final", "sweeps", "levels", "capped"))
    return s


def _summary(r):
    return {"best_spins": r.best_spins, "best_energy": float(r.best_energy), "best_replica": int(r.best_replica),
            "mean_energy": float(r.mean_energy), "sweeps": int(r.sweeps), "levels": int(r.levels), "hits": int(r.hits)}


def run(state):
    ctx, case = state.ctx, state.case
    if state.kind == "batch":
        return [_summary(r) for r in ctx.solve_batch(state.jobs)]
    if state.kind == "serve":
        reqs = [ctx.submit(inst, R, 0.0, t_max, c_step=c, seed=sd, precision=prec,
                           fixed_sweeps=4 if prec == "bf16" else 0)
                for (inst, t_max, c, prec), R, sd in state.requests]
        done, pending = {}, list(reqs)
        while pending:
            for q in list(pending):
                r = ctx.poll(q)
                if r is not None:
                    done[q] = r
                    pending.remove(q)
            if pending:
                time.sleep(0.0002)
        return {"best_spins": np.concatenate([done[q].best_spins for q in reqs]),
                "best_energy": np.array([done[q].best_energy for q in reqs]),
                "mean_energy": np.array([done[q].mean_energy for q in reqs]),
                "sweeps": np.array([done[q].sweeps for q in reqs])}
    if state.kind == "energy":
        e, ei = ctx.energy(state.inst, state.spins)
        return {"e": e, "e_i64": ei}
    r = ctx.solve(state.inst, case["replicas"], 0.0, case["t_max"], **state.kw)
    out = _summary(r)
    for k in state.kw["outputs"]:
        out["replica_" + k] = getattr(r, {"sweeps": "replica_sweeps", "levels": "replica_levels",
                                          "capped": "replica_capped"}.get(k, k))
    return out


def _pairs(case):
    """Stored couplings (both directions) of one instance, and its spins."""
    if case["family"].startswith("sk_"):
        return case["size"] * (case["size"] - 1), case["size"]
    if case["family"] == "ea":
        return 2 * case["dim"] * case["size"] ** case["dim"], case["size"] ** case["dim"]
    return case["size"] * case["degree"], case["size"]


def work(case):
    """What a pass cannot do without. Sweeps under the stopping rule are counted
    as 8 per level, the least that converging levels take; a replica visits half
    of the levels on average. A sweep needs 2 flops per stored coupling and spin;
    bytes are the couplings and the outputs once."""
    if case["kind"] == "batch":
        n, R = case["size"], case["replicas"]
        return {"bytes": float(case["jobs"] * (24 * n * 4 + n * R // 2)),
                "flops": float(case["jobs"] * 2 * 24 * 0.7 * n * (R / 2) * 8 * 6)}
    if case["kind"] == "serve":
        n, R = 16 * case["size"], case["replicas"] // 2
        return {"bytes": float(case["requests"] * (12 * n * 4 + n)),
                "flops": float(case["requests"] * 2 * 12 * n * R * 8 * 4)}
    nnz, n = _pairs(case)
    dense = case["family"].startswith("sk_")
    width = 1 if case["family"] == "sk_pm1" else 4
    if case["kind"] == "energy":
        return {"bytes": float(nnz * width + case["count"] * (n + 16)), "flops": float(case["count"] * nnz)}
    R = case["replicas"]
    per = case["sweeps"] if case["sweeps"] else 8
    sweeps = R * max(1.0, case["levels"] / 2) * per
    couplings = nnz * ({"fp32": width, "bf16": 2, "fp8": 1}[case["precision"]] if dense else 4)
    outputs = R * n * 4 + (R * n if case["sweeps"] and case["method"] == "mars" else 0) + n + 20 * R
    if not dense and n > 55000:  # the replicas' state streams through HBM
        couplings += 12.0 * n * sweeps
    return {"bytes": float(couplings + outputs), "flops": 2.0 * nnz * sweeps}


def _philox(c0, c1, c2, c3, seed):
    """Words 0 and 1 of Philox4x32-10 at tensors of counters (int64)."""
    mask = 0xFFFFFFFF
    k0, k1 = seed & mask, (seed >> 32) & mask
    c = [torch.as_tensor(x, dtype=torch.int64, device="cuda") for x in (c0, c1, c2, c3)]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c[0], c[1]


def _nmfa_exact(case, seed):
    """Noisy mean-field annealing as the library documents it, in float64."""
    n, R = case["size"], case["replicas"]
    if case["family"] == "er":
        J = torch.from_numpy(instances.csr_to_dense(_sparse(case, seed))).cuda()
    else:
        J = _dense(case, seed).double()
    m0, t0 = _start(case, seed)
    s, T = m0.double(), t0.double()
    norm = J.square().sum(1).sqrt()
    inv = torch.where(norm > 0, 1.0 / norm.clamp_min(1e-300), torch.zeros_like(norm))
    i = torch.arange(n, dtype=torch.int64, device="cuda")[None, :]
    r = torch.arange(R, dtype=torch.int64, device="cuda")[:, None]
    k = 0
    while True:
        T = T - case["t_max"] / case["levels"]
        live = T > 0
        if not bool(live.any()):
            break
        w0, w1 = _philox((i >> 1).expand(R, n), r.expand(R, n), torch.full((R, n), 2 + k, device="cuda"),
                         torch.zeros((R, n), device="cuda"), seed)
        u1, u2 = ((w0 >> 8) + 1).double() * 2.0 ** -24, (w1 >> 8).double() * 2.0 ** -24
        ang = 2.0 * math.pi * u2
        xi = (-2.0 * u1.log()).sqrt() * torch.where((i & 1) == 1, ang.sin(), ang.cos())
        shat = -torch.tanh(((s @ J) * inv + 0.15 * xi) / T.clamp_min(1e-300)[:, None])
        s = torch.where(live[:, None], 0.5 * shat + 0.5 * s, s)
        k += 1
    sg = torch.where(s >= 0, 1.0, -1.0).double()
    e = 0.5 * ((sg @ J) * sg).sum(1)
    return {"best_spins": None, "best_energy": None, "best_replica": None, "mean_energy": None, "sweeps": None,
            "levels": None, "hits": None, "replica_energies": e, "replica_m_final": s}


def exact(case, seed):
    if case["kind"] == "solve" and case["method"] == "nmfa":
        return _nmfa_exact(case, seed)
    if case["kind"] != "energy":
        return None  # see the module's docstring
    sp = torch.from_numpy(_spins(case, seed)).cuda().double()
    if case["family"] == "er":
        rp, col, val = _sparse(case, seed)
        rows = torch.from_numpy(np.repeat(np.arange(case["size"]), np.diff(rp))).cuda()
        cols, v = torch.from_numpy(col).cuda().long(), torch.from_numpy(val).cuda()
        e = torch.stack([0.5 * (v * x[rows] * x[cols]).sum() for x in sp])
    else:
        e = 0.5 * ((sp @ _dense(case, seed).double()) * sp).sum(1)
    return {"e": e, "e_i64": None}
