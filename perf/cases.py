"""The work this framework is used for, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` gives the standing cases and
``draw(rng)`` one more from the same ranges; ``prepare(case, seed)`` makes what
a program holds before the call, ``run(state)`` is one pass through the public
entry points, ``work(case)`` the bytes and operations of a pass that no
implementation can do without, and ``exact(case, seed)`` the first pass's
outputs in 64 bits by plain torch and numpy.

Inputs: density 3 per r_c^3, alpha = 4, dt = 0.01, the positions of a sheared
run past its first few hundred steps.  There the particles cluster: ~18
partners per row with a standard deviation of ~8 and S(q -> 0) ~ 20, which the
density field of ``_positions`` reproduces (a log-normal field of correlation
length ~r_c, consistent with the Lees-Edwards images).
"""
import math
import random

import numpy as np
import torch

import paper_1808_06381_gb300 as ss

DENSITY, ALPHA, DT, RC = 3.0, 4.0, 0.01, 1.0
LAMBDA2 = RC * RC / (2.0 * math.log(20.0))   # the pair weight is 5 % at r_c
C_EV = 0.1 / LAMBDA2                         # excluded volume, eps = kT = 1
NOISE = math.sqrt(2.0 / DT)                  # zeta = kT = 1
PAIRS = 18.0                                 # partners per particle
ITERATIONS = 45.0                            # CG iterations to 1e-8
CUBE = (1.0, 1.0, 1.0)
PAPER = (35.79, 17.81, 8.99)                 # edges of the box of the velocity-correlation figure


def listed():
    return [
        # the smallest call: one step of a few hundred particles, all latency
        {"name": "step-fp64-n500", "kind": "step", "n": 500, "precision": "fp64", "kappa_tau": 0.5, "tol": 1e-10, "nsteps": 1},
        # the plain FP64 workload, ten steps between two frames read back
        {"name": "run-fp64-n4096", "kind": "step", "n": 4096, "precision": "fp64", "kappa_tau": 0.5, "tol": 1e-10, "nsteps": 10},
        # an FP64 reference step of a mid-sized ragged system
        {"name": "step-fp64-n60013", "kind": "step", "n": 60013, "precision": "fp64", "kappa_tau": 0.5, "tol": 1e-8, "nsteps": 1},
        # a small production run at low shear, mixed precision
        {"name": "run-mixed-n20011", "kind": "step", "n": 20011, "precision": "mixed", "kappa_tau": 0.05, "tol": 1e-8, "nsteps": 4},
        # the default workload: one step from and to host positions, the solver tuned once
        {"name": "step-mixed-n262144", "kind": "step", "n": 262144, "precision": "mixed", "kappa_tau": 0.5, "tol": 1e-8, "nsteps": 1, "tune": True},
        # the large-scale workload, bound by HBM
        {"name": "step-mixed-n4194304", "kind": "step", "n": 4194304, "precision": "mixed", "kappa_tau": 0.5, "tol": 1e-8, "nsteps": 1, "tune": True},
        # an ensemble advanced together: sizes and shear rates spread as in the replica workload
        {"name": "batch-8", "kind": "batch", "replicas": 8, "mix": 1, "lo": 8192, "hi": 131072, "tol": 1e-8},
        # the velocity cross-correlation of a frame, the paper's box, 120 bins to 30 lambda
        {"name": "vcorr-n17191", "kind": "vcorr", "n": 17191, "paper_box": True, "nbins": 120, "rmax_lambda": 30.0, "kappa_tau": 0.0},
        # S(qx, qy) of the current configuration on the grid that the large workload uses
        {"name": "sfactor-n262144", "kind": "sfactor", "n": 262144, "nk": 48, "grid": 256},
        # A^(1/2) g of the default system: thermal noise consistent with the friction
        {"name": "sqrt-n262144", "kind": "sqrt", "n": 262144, "precision": "mixed", "degree": 32},
        # one optimiser step of the learned warm start on the system just solved
        {"name": "train-n262144", "kind": "train", "n": 262144},
        # the allocation-free solve of a caller's own CSR system
        {"name": "csr-n12289", "kind": "csr", "n": 12289, "tol": 1e-10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["step64", "mixed", "mixed", "batch", "vcorr", "sfactor", "sqrt", "train", "csr"])
    if kind == "step64":
        n = _log(rng, 300, 200000)
        return {"kind": "step", "n": n, "precision": "fp64", "kappa_tau": round(rng.uniform(0.05, 1.0), 3),
                "tol": rng.choice([1e-8, 1e-10]), "nsteps": rng.randint(1, 10) if n < 8000 else 1}
    if kind == "mixed":
        n = _log(rng, 1000, 4000000)
        return {"kind": "step", "n": n, "precision": "mixed", "kappa_tau": round(rng.uniform(0.05, 1.0), 3),
                "tol": 1e-8, "nsteps": rng.randint(1, 4) if n < 30000 else 1, "tune": rng.random() < 0.5}
    if kind == "batch":
        lo = _log(rng, 2000, 20000)
        return {"kind": "batch", "replicas": rng.randint(2, 12), "mix": rng.randint(0, 10 ** 6), "lo": lo, "hi": lo * rng.choice([2, 4, 8]), "tol": 1e-8}
    if kind == "vcorr":
        n = _log(rng, 500, 40000)
        return {"kind": "vcorr", "n": n, "paper_box": False, "nbins": rng.randint(10, 300),
                "rmax_lambda": round(rng.uniform(0.15, 0.6) * (n / DENSITY) ** (1 / 3) / math.sqrt(LAMBDA2), 2),
                "kappa_tau": rng.choice([0.0, 0.5])}
    if kind == "sfactor":
        grid = rng.choice([0, 64, 128, 256, 512])
        return {"kind": "sfactor", "n": _log(rng, 2000, 40000 if grid == 0 else 1000000),
                "nk": rng.randint(2, 12 if grid == 0 else min(64, grid // 4 - 1)), "grid": grid}
    if kind == "sqrt":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        return {"kind": "sqrt", "n": _log(rng, 1000, 400000), "precision": precision, "degree": rng.randint(8, 64)}
    if kind == "train":
        return {"kind": "train", "n": _log(rng, 3000, 400000)}
    return {"kind": "csr", "n": _log(rng, 300, 32768), "tol": rng.choice([1e-8, 1e-10])}


# ---------------------------------------------------------------- inputs

def _positions(n, L, delta, seed):
    """n clustered positions in [0, L), float64 [n, 3] on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    Lt = torch.tensor(L, dtype=torch.float64, device="cuda")
    modes, sigma, length = 64, 0.72, 0.95
    m = torch.round(torch.randn(modes, 3, generator=g, device="cuda", dtype=torch.float64) / length * Lt / (2 * math.pi))
    k = 2 * math.pi * m / Lt
    k[:, 1] -= delta / L[1] * k[:, 0]   # the reciprocal lattice of the sheared box
    phase = 2 * math.pi * torch.rand(modes, generator=g, device="cuda", dtype=torch.float64)
    kf, ph = k.float().T.contiguous(), phase.float()
    got, have = [], 0
    while have < n:
        c = min(1 << 20, 2048 + 6 * (n - have))
        x = torch.rand(c, 3, generator=g, device="cuda", dtype=torch.float64) * Lt
        f = math.sqrt(2.0 / modes) * torch.cos(x.float() @ kf + ph).sum(1)
        keep = torch.rand(c, generator=g, device="cuda") < torch.exp(sigma * (f - 2.5))
        x = x[keep]
        got.append(x)
        have += x.shape[0]
    pos = torch.cat(got)[:n]
    return torch.where(pos >= Lt, torch.zeros_like(pos), pos).contiguous()


def _frame(n, seed, edges=None):
    """(L, image offset, positions) of one configuration."""
    L = tuple(edges) if edges else ((n / DENSITY) ** (1.0 / 3.0),) * 3
    delta = random.Random(seed).uniform(0.0, 0.999) * L[0]
    return L, delta, _positions(n, L, delta, seed)


def _pinned(n):
    return torch.empty((n, 3), dtype=torch.float64, pin_memory=True)


def _kappa(kappa_tau):
    return kappa_tau / LAMBDA2


def _replicas(case, seed):
    """(n, kappa tau, seed) of every replica: sizes and rates of the ensemble, log-uniform."""
    rng = random.Random(case["mix"])
    return [(_log(rng, case["lo"], case["hi"]), math.exp(rng.uniform(math.log(0.01), 0.0)), seed * 100 + r)
            for r in range(case["replicas"])]


def _vcorr_inputs(case, seed):
    L, delta, pos = _frame(case["n"], seed, PAPER if case["paper_box"] else None)
    kappa = _kappa(case["kappa_tau"])
    if kappa == 0.0:
        delta = 0.0
    # velocities of the last solve: a flow that neighbours share, thermal noise, the shear
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    Lt = torch.tensor(L, dtype=torch.float64, device="cuda")
    k = 2 * math.pi / Lt * torch.randint(-6, 7, (12, 3), generator=g, device="cuda")
    amp = torch.randn(12, 3, generator=g, device="cuda", dtype=torch.float64)
    v = torch.cos(pos @ k.T) @ amp * 0.5 + 1.5 * torch.randn(pos.shape, generator=g, device="cuda", dtype=torch.float64)
    v[:, 0] += kappa * (pos[:, 1] - 0.5 * L[1])
    return L, delta, kappa, pos, v, case["rmax_lambda"] * math.sqrt(LAMBDA2)


def _simulation(case, seed, L, precision, pos, kappa_tau=0.5, tol=1e-8, warm="prev"):
    return ss.Simulation(case["n"], L, _kappa(kappa_tau), alpha=ALPHA, dt=DT, seed=seed, precision=precision,
                         warm_start=warm, cg_tol=tol, positions=pos.cpu().numpy())


def _weights(seed):
    """Weights of the network part way through training: scaled normals, a mixed readout."""
    r = np.random.Generator(np.random.PCG64(seed))
    return np.concatenate([r.normal(0, 6 ** -0.5, 6 * 64), r.normal(0, 0.125, 64 * 64), r.normal(0, 0.125, 64 * 4),
                           r.normal(0, 0.6, 11)]).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        L, delta, pos = _frame(case["n"], seed)
        sim = _simulation(case, seed, L, case["precision"], pos, case["kappa_tau"], case["tol"])
        pos_in, pos_out = _pinned(case["n"]), _pinned(case["n"])
        pos_in.copy_(pos)
        if case.get("tune"):
            sim.autotune(trials=1)
        sim.step_host(pos_in.numpy(), delta, 0, pos_out.numpy())   # the handle of a running program: step graph captured
        return {"kind": kind, "sim": sim, "delta": delta, "in": pos_in, "out": pos_out, "nsteps": case["nsteps"]}
    if kind == "batch":
        reps, frames = _replicas(case, seed), []
        for n, _, s in reps:
            frames.append(_frame(n, s))
        batch = ss.Batch([{"n": n, "L": f[0], "kappa": _kappa(kt), "alpha": ALPHA, "dt": DT, "seed": s, "cg_tol": case["tol"]}
                          for (n, kt, s), f in zip(reps, frames)], positions=[f[2].cpu().numpy() for f in frames])
        sims = [batch.sim(r) for r in range(len(reps))]
        return {"kind": kind, "batch": batch, "sims": sims, "out": [_pinned(n) for n, _, _ in reps]}
    if kind == "vcorr":
        L, delta, kappa, pos, v, rmax = _vcorr_inputs(case, seed)
        return {"kind": kind, "args": (pos.cpu().numpy(), v.cpu().numpy(), L, delta, kappa, case["nbins"], rmax)}
    if kind == "csr":
        L, delta, pos = _frame(case["n"], seed)
        s = _system(pos, L, delta, _kappa(0.5), seed, 0)
        crow, col = s["crow"].int().contiguous(), s["j"].int().contiguous()
        return {"kind": kind, "n": case["n"], "tol": case["tol"], "crow": crow, "col": col, "w": s["w"], "diag": s["diag"],
                "b": s["b"].T.contiguous(), "x": torch.zeros(3, case["n"], dtype=torch.float64, device="cuda")}
    L, delta, pos = _frame(case["n"], seed)
    sim = _simulation(case, seed, L, case.get("precision", "mixed"), pos)
    sim.set_positions(pos.cpu().numpy(), delta)
    if kind == "sfactor":
        return {"kind": kind, "sim": sim, "nk": case["nk"], "grid": case["grid"]}
    sim.build_neighbors()
    sim.assemble()
    if kind == "sqrt":
        g = np.random.Generator(np.random.PCG64(seed)).standard_normal((case["n"], 3))
        return {"kind": kind, "sim": sim, "g": g, "degree": case["degree"]}
    sim.solve_velocities()                    # the previous step's velocities, a feature of the network
    sim.mpnn_enable(weights=_weights(seed))
    sim.set_step(1)
    sim.assemble()
    sim.mpnn_forward()
    sim.solve_velocities()                    # the target
    return {"kind": kind, "sim": sim}


def run(state):
    kind = state["kind"]
    if kind == "step":
        info = state["sim"].step_host(state["in"].numpy(), state["delta"], state["nsteps"], state["out"].numpy())
        return {"pos": state["out"], "stress": info["stress_xy"]}
    if kind == "batch":
        infos = state["batch"].step(1)
        for sim, out in zip(state["sims"], state["out"]):
            sim.get_positions(out.numpy())
        return {"pos": state["out"], "stress": [i["stress_xy"] for i in infos]}
    if kind == "vcorr":
        r = ss.velocity_correlation(*state["args"])
        return {key: r[key] for key in ("sums", "counts", "vsq", "correlation")}
    if kind == "sfactor":
        S, qx, qy = state["sim"].structure_factor(state["nk"], state["nk"], grid=state["grid"])
        return {"S": S, "qx": qx, "qy": qy}
    if kind == "sqrt":
        xi, lmax = state["sim"].sqrt_apply(state["g"], state["degree"])
        return {"xi": xi, "lmax": lmax}
    if kind == "train":
        loss, grad = state["sim"].mpnn_train_step(lr=2e-3, want_grad=True)
        return {"loss": loss, "grad": grad}
    stream = torch.cuda.current_stream().cuda_stream
    info = ss.solve_csr_noalloc(state["n"], state["crow"].data_ptr(), state["col"].data_ptr(), state["w"].data_ptr(),
                                state["diag"].data_ptr(), ALPHA, state["b"].data_ptr(), state["x"].data_ptr(),
                                tol=state["tol"], max_iter=1000, stream=stream)
    if info["status"] != ss.SP_OK:
        raise RuntimeError(info["error"])
    return {"x": state["x"]}


def work(case):
    """Bytes: inputs read once and outputs written once; flops: the pair terms, the
    solver's products (6 per stored entry and iteration) and vector updates (30 per row)."""
    kind, n = case["kind"], float(case.get("n", 0))
    solve = ITERATIONS * (6.0 * PAIRS + 30.0)
    step = 60.0 * PAIRS + solve
    if kind == "step":
        return {"bytes": 48.0 * n, "flops": step * n * case["nsteps"]}
    if kind == "batch":
        n = float(sum(r[0] for r in _replicas(case, 0)))
        return {"bytes": 48.0 * n, "flops": step * n}
    if kind == "vcorr":
        return {"bytes": 48.0 * n + 16.0 * case["nbins"], "flops": 22.0 * 0.5 * n * n}
    if kind == "sfactor":
        modes = (2.0 * case["nk"] + 1) ** 2
        if case["grid"] == 0:
            return {"bytes": 16.0 * n + 24.0 * modes, "flops": 8.0 * n * modes}
        G = float(case["grid"])
        return {"bytes": 16.0 * n + 24.0 * modes, "flops": 20.0 * n + 10.0 * G * G * math.log2(G)}
    if kind == "sqrt":
        return {"bytes": 48.0 * n + 12.0 * PAIRS * n, "flops": case["degree"] * (6.0 * PAIRS + 24.0) * n}
    if kind == "train":   # three rows per particle: forward again, two activation and three weight products
        mac = 2 * (6 * 64 + 64 * 64) + 64 * 4 + (64 * 64 + 64 * 4) + 8 * PAIRS / 3
        return {"bytes": (3 * 16.0 * 3 + 12.0 + 8.0 * PAIRS) * n, "flops": 2.0 * 3 * n * mac}
    return {"bytes": (12.0 * PAIRS + 60.0) * n, "flops": solve * n}


# ---------------------------------------------------------------- 64-bit reference

def _pairs(pos, L, delta):
    """Directed pairs (i, j, R_i - R_j, y image) within r_c, ordered by i, on the sheared box."""
    n, dev = pos.shape[0], pos.device
    reach = RC * 1.0001
    up, down = pos[:, 1] < reach, pos[:, 1] > L[1] - reach
    ids = torch.arange(n, device=dev)
    ghost, gid, gm = [pos], [ids], [torch.zeros(n, dtype=torch.float64, device=dev)]
    for sel, m in ((up, 1.0), (down, -1.0)):   # the image m boxes up lies at x + m delta
        q = pos[sel].clone()
        q[:, 0] = torch.remainder(q[:, 0] + m * delta, L[0])
        q[:, 1] += m * L[1]
        ghost.append(q)
        gid.append(ids[sel])
        gm.append(torch.full((q.shape[0],), m, dtype=torch.float64, device=dev))
    q, gid, gm = torch.cat(ghost), torch.cat(gid), torch.cat(gm)
    nc = [max(1, int(L[a] / (RC * 1.001))) for a in range(3)]
    ny = nc[1] + 4

    def cells(p):
        cx = (p[:, 0] * (nc[0] / L[0])).long().clamp(0, nc[0] - 1)
        cy = torch.floor(p[:, 1] * (nc[1] / L[1])).long() + 2
        cz = (p[:, 2] * (nc[2] / L[2])).long().clamp(0, nc[2] - 1)
        return cx, cy, cz

    cx, cy, cz = cells(q)
    cell = (cz * ny + cy) * nc[0] + cx
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=nc[0] * ny * nc[2])
    start = torch.cumsum(count, 0) - count
    q, gid, gm = q[order], gid[order], gm[order]
    cx, cy, cz = cells(pos)
    rows, cols, seps, images = [], [], [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                c = ((cz + dz) % nc[2] * ny + cy + dy) * nc[0] + (cx + dx) % nc[0]
                s, cnt = start[c], count[c]
                for k in range(int(cnt.max())):
                    i = torch.nonzero(cnt > k).squeeze(1)
                    at = s[i] + k
                    d = pos[i] - q[at]
                    d[:, 0] -= L[0] * torch.round(d[:, 0] / L[0])
                    d[:, 2] -= L[2] * torch.round(d[:, 2] / L[2])
                    ok = ((d * d).sum(1) < RC * RC) & (gid[at] != i)
                    if bool(ok.any()):
                        rows.append(i[ok])
                        cols.append(gid[at][ok])
                        seps.append(d[ok])
                        images.append(gm[at][ok])
    i, j, d, m = torch.cat(rows), torch.cat(cols), torch.cat(seps), torch.cat(images)
    order = torch.argsort(i, stable=True)
    return i[order], j[order], d[order], m[order]


def _normals(seed, step, n):
    """Box-Muller normals of Philox4x64-10 blocks with key (seed, 0), counter (id, step, 0, 0)."""
    first = ((step << 64) - 1) % (1 << 256)   # numpy advances the counter before each block
    words = np.array([(first >> (64 * k)) % (1 << 64) for k in range(4)], dtype=np.uint64)
    raw = np.random.Philox(key=np.array([seed, 0], dtype=np.uint64), counter=words).random_raw(4 * n).reshape(n, 4)
    u = torch.from_numpy(((raw >> np.uint64(11)).astype(np.float64) + [1.0, 0.0, 1.0, 0.0]) * 2.0 ** -53).cuda()
    r1, r2 = torch.sqrt(-2.0 * torch.log(u[:, 0])), torch.sqrt(-2.0 * torch.log(u[:, 2]))
    a, b = 2 * math.pi * u[:, 1], 2 * math.pi * u[:, 3]
    return torch.stack([r1 * torch.cos(a), r1 * torch.sin(a), r2 * torch.cos(b)], 1)


def _system(pos, L, delta, kappa, seed, step):
    """(I + alpha L_w) v = b of one configuration, with its pairs."""
    n = pos.shape[0]
    i, j, d, m = _pairs(pos, L, delta)
    w = torch.exp(-(d * d).sum(1) / (2.0 * LAMBDA2))
    crow = torch.zeros(n + 1, dtype=torch.long, device=pos.device)
    crow[1:] = torch.cumsum(torch.bincount(i, minlength=n), 0)
    per_row = lambda x: torch.segment_reduce(x, "sum", offsets=crow, axis=0, initial=0)   # noqa: E731
    b = NOISE * _normals(seed, step, n) + C_EV * per_row(d * w[:, None])
    b[:, 0] += kappa * (pos[:, 1] - 0.5 * L[1]) + ALPHA * kappa * L[1] * per_row(m * w)
    return {"i": i, "j": j, "d": d, "m": m, "w": w, "crow": crow, "diag": 1.0 + ALPHA * per_row(w), "b": b}


def _matrix(s):
    n = s["diag"].shape[0]
    return torch.sparse_csr_tensor(s["crow"].int(), s["j"].int(), s["w"], size=(n, n))


def _solve(s, tol=1e-13):
    """Jacobi-preconditioned conjugate gradients."""
    W, D, b = _matrix(s), s["diag"][:, None], s["b"]
    apply = lambda u: D * u - ALPHA * (W @ u)   # noqa: E731
    x = torch.zeros_like(b)
    r, stop = b.clone(), tol * float(b.norm())
    z = r / D
    p, rho = z.clone(), (r * z).sum()
    for _ in range(2000):
        q = apply(p)
        a = rho / (p * q).sum()
        x += a * p
        r -= a * q
        if float(r.norm()) <= stop:
            break
        z = r / D
        new = (r * z).sum()
        p = z + new / rho * p
        rho = new
    return x


def _exact_steps(pos, L, delta, kappa, seed, nsteps):
    for step in range(nsteps):
        s = _system(pos, L, delta, kappa, seed, step)
        v = _solve(s)
        f = C_EV * s["d"][:, 0] * s["w"] + ALPHA * s["w"] * (v[s["j"], 0] - v[s["i"], 0] + kappa * L[1] * s["m"])
        stress = -0.5 * float((s["d"][:, 1] * f).sum()) / (L[0] * L[1] * L[2])
        delta = math.fmod(delta + kappa * L[1] * DT, L[0])
        pos = pos + v * DT
        for off, sign in ((pos[:, 1] < 0.0, 1.0), (pos[:, 1] >= L[1], -1.0)):
            pos[:, 1] = torch.where(off, pos[:, 1] + sign * L[1], pos[:, 1])
            pos[:, 0] = torch.where(off, pos[:, 0] + sign * delta, pos[:, 0])
        for a in (0, 2):
            pos[:, a] -= L[a] * torch.floor(pos[:, a] / L[a])
    return pos, stress


def _exact_vcorr(case, seed):
    L, delta, kappa, pos, v, rmax = _vcorr_inputs(case, seed)
    n, nbins = case["n"], case["nbins"]
    u = v.clone()
    u[:, 0] -= kappa * (pos[:, 1] - 0.5 * L[1])
    away = lambda x: torch.sign(x) * torch.floor(x.abs() + 0.5)   # noqa: E731  (half away from zero)
    sums = torch.zeros(nbins, dtype=torch.float64, device="cuda")
    counts = torch.zeros(nbins, dtype=torch.long, device="cuda")
    for a in range(0, n, 512):
        d = pos[a:a + 512, None, :] - pos[None, a:, :]
        m = away(d[..., 1] / L[1])
        dy = d[..., 1] - m * L[1]
        dx = d[..., 0] - m * delta
        dx = dx - L[0] * away(dx / L[0])
        dz = d[..., 2] - L[2] * away(d[..., 2] / L[2])
        r2 = dx * dx + dy * dy + dz * dz
        ok = (r2 < rmax * rmax) & (torch.arange(a, n, device="cuda")[None, :] > torch.arange(a, min(n, a + 512), device="cuda")[:, None])
        k = torch.floor(torch.sqrt(r2[ok]) * (nbins / rmax)).long().clamp(max=nbins - 1)
        sums.index_add_(0, k, (u[a:a + 512] @ u[a:].T)[ok])
        counts += torch.bincount(k, minlength=nbins)
    vsq = float((u * u).sum()) / n
    return {"sums": sums, "counts": counts, "vsq": vsq, "correlation": sums / (counts * vsq)}


def _exact_sfactor(case, seed):
    n, nk, G = case["n"], case["nk"], case["grid"]
    L, delta, pos = _frame(n, seed)
    k = torch.arange(-nk, nk + 1, dtype=torch.float64, device="cuda")
    qx = (2 * math.pi / L[0] * k)[:, None].expand(2 * nk + 1, 2 * nk + 1)
    qy = 2 * math.pi / L[1] * k[None, :] - delta / L[1] * qx
    if G == 0:
        S = torch.empty(2 * nk + 1, 2 * nk + 1, dtype=torch.float64, device="cuda")
        for a in range(2 * nk + 1):
            ph = pos[:, :1] * qx[a] + pos[:, 1:2] * qy[a]
            S[a] = (torch.cos(ph).sum(0) ** 2 + torch.sin(ph).sum(0) ** 2) / n
        return {"S": S, "qx": qx, "qy": qy}
    # cloud-in-cell density in the sheared frame, its transform, the window divided out
    xs = pos[:, 0] - delta / L[1] * pos[:, 1]
    xs = (xs - L[0] * torch.floor(xs / L[0])) / L[0] * G
    ys = pos[:, 1] / L[1] * G
    i0, j0 = torch.floor(xs).long(), torch.floor(ys).long()
    fx, fy = xs - i0, ys - j0
    rho = torch.zeros(G * G, dtype=torch.float64, device="cuda")
    for di, wx in ((0, 1 - fx), (1, fx)):
        for dj, wy in ((0, 1 - fy), (1, fy)):
            rho.index_add_(0, (j0 + dj) % G * G + (i0 + di) % G, wx * wy)
    F = torch.fft.fft2(rho.reshape(G, G))
    at = torch.arange(-nk, nk + 1, device="cuda") % G
    F = F[at][:, at].T
    win = torch.sinc(k / G) ** 2
    return {"S": F.abs() ** 2 / (win[:, None] * win[None, :]) ** 2 / n, "qx": qx, "qy": qy}


def _exact_sqrt(case, seed):
    L, delta, pos = _frame(case["n"], seed)
    s = _system(pos, L, delta, 0.0, seed, 0)
    W, D = _matrix(s), s["diag"][:, None]
    lmax = float((2 * s["diag"] - 1).max())
    N = case["degree"] + 1
    th = math.pi * (np.arange(N) + 0.5) / N
    c = 2.0 / N * (np.sqrt(0.5 * (lmax - 1) * np.cos(th) + 0.5 * (lmax + 1)) * np.cos(np.arange(N)[:, None] * th)).sum(1)
    u = lambda t: (2 * (D * t - ALPHA * (W @ t)) - (lmax + 1) * t) / (lmax - 1)   # noqa: E731
    t0 = torch.from_numpy(np.random.Generator(np.random.PCG64(seed)).standard_normal((case["n"], 3))).cuda()
    t1 = u(t0)
    xi = 0.5 * c[0] * t0 + c[1] * t1
    for k in range(2, N):
        t0, t1 = t1, 2 * u(t1) - t0
        xi += c[k] * t1
    return {"xi": xi, "lmax": lmax}


def _exact_train(case, seed):
    """Loss and gradient of the network (no rounding to 16 bits)."""
    n = case["n"]
    L, delta, pos = _frame(n, seed)
    vprev = _solve(_system(pos, L, delta, _kappa(0.5), seed, 0))
    s = _system(pos, L, delta, _kappa(0.5), seed, 1)
    W, D, b = _matrix(s), s["diag"][:, None], s["b"]
    w = torch.from_numpy(_weights(seed).astype(np.float64)).cuda()
    W1, W2, W3, o = w[:384].view(6, 64), w[384:4480].view(64, 64), w[4480:4736].view(64, 4), w[4736:]
    M = lambda x: (ALPHA * (W @ x.reshape(n, -1)) / D).reshape(3 * n, -1)   # noqa: E731
    MT = lambda x: (ALPHA * (W @ (x.reshape(n, -1) / D))).reshape(3 * n, -1)   # noqa: E731
    scale = float((b * b).sum() / (3 * n)) ** 0.5
    x0 = torch.stack([b / D, vprev, b], 2).reshape(3 * n, 3) / scale
    inp = torch.cat([x0, M(x0)], 1)
    h1 = torch.tanh(inp @ W1)
    h2 = torch.tanh(h1 @ W2)
    y = h2 @ W3
    feat = torch.cat([y, M(y), x0], 1)
    e = feat @ o - _solve(s).reshape(3 * n) / scale
    d = 2 * e / (3 * n)
    dy = d[:, None] * o[:4] + MT(d[:, None] * o[4:8])
    p2 = dy @ W3.T * (1 - h2 * h2)
    p1 = p2 @ W2.T * (1 - h1 * h1)
    grad = torch.cat([(inp.T @ p1).ravel(), (h1.T @ p2).ravel(), (h2.T @ dy).ravel(), feat.T @ d])
    return {"loss": float((e * e).sum() / (3 * n)), "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        L, delta, pos = _frame(case["n"], seed)
        pos, stress = _exact_steps(pos, L, delta, _kappa(case["kappa_tau"]), seed, case["nsteps"])
        return {"pos": pos, "stress": stress}
    if kind == "batch":
        out = []
        for n, kt, s in _replicas(case, seed):
            L, _, pos = _frame(n, s)
            out.append(_exact_steps(pos, L, 0.0, _kappa(kt), s, 1))   # a batch starts with offset 0
        return {"pos": [p for p, _ in out], "stress": [t for _, t in out]}
    if kind == "vcorr":
        return _exact_vcorr(case, seed)
    if kind == "sfactor":
        return _exact_sfactor(case, seed)
    if kind == "sqrt":
        return _exact_sqrt(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    L, delta, pos = _frame(case["n"], seed)
    return {"x": _solve(_system(pos, L, delta, _kappa(0.5), seed, 0)).T.contiguous()}
