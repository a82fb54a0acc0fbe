"""What a program asks of this engine, as measurable cases.

Every case is one call (or one short session) through the public Python entry points over a
synthetic system shaped like the configurations of this repository: water boxes, fcc crystals and
the solvated-chain mixture, F = 64 or 128, three layers, 20 Gaussians, cutoff 5 A, in FP32 and on
the BF16 path, from a 192-atom box to the 1,000,188-atom crystal.

The engine returns double arrays whatever the precision of the path; a caller that asked for the
FP32 or BF16 path keeps them in that precision, and so do the cases: FP32 results in float32, BF16
results in bfloat16.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2506_04055_gb300 as eng
import synthetic as syn

RC = 5.0
DEV = "cuda"
ACC = 9.648533212331002e-3   # A / fs^2 per eV / A / amu


def listed():
    return [
        # the smallest system of the repository's configurations: call latency
        {"name": "water_192_fp32", "kind": "call", "system": "water", "n": 192, "F": 64, "T": 3, "K": 20,
         "precision": "fp32", "rebuild": False},
        # a unit-cell-sized crystal on the tensor-core path, the small end of a screening run
        {"name": "fcc_500_bf16", "kind": "call", "system": "fcc", "n": 500, "F": 128, "T": 3, "K": 20,
         "precision": "bf16", "rebuild": False},
        # a single point on a new geometry: the neighbour list is built in the call
        {"name": "water_6k_rebuild_fp32", "kind": "call", "system": "water", "n": 5997, "F": 64, "T": 3, "K": 20,
         "precision": "fp32", "rebuild": True},
        # the 96,000-atom water box inside an MD code that keeps its own integrator, both precisions
        {"name": "water_96k_fp32", "kind": "call", "system": "water", "n": 96000, "F": 64, "T": 3, "K": 20,
         "precision": "fp32", "rebuild": False},
        {"name": "water_96k_bf16", "kind": "call", "system": "water", "n": 96000, "F": 64, "T": 3, "K": 20,
         "precision": "bf16", "rebuild": False},
        # a mid-sized crystal at the wide model, FP32
        {"name": "fcc_32k_fp32", "kind": "call", "system": "fcc", "n": 32000, "F": 128, "T": 3, "K": 20,
         "precision": "fp32", "rebuild": False},
        # the headline workload: 63^3 fcc cells, BF16
        {"name": "fcc_1m_bf16", "kind": "call", "system": "fcc", "n": 1000188, "F": 128, "T": 3, "K": 20,
         "precision": "bf16", "rebuild": False},
        # differentiation of the energy by the autograd Function on the triclinic mixture
        {"name": "mixture_90k_grad_fp32", "kind": "grad", "system": "mixture", "n": 90300, "F": 64, "T": 2, "K": 20,
         "precision": "fp32"},
        # the strictly local family, both precisions
        {"name": "local_12k_fp32", "kind": "local", "system": "water", "n": 12000, "F": 64, "T": 2, "K": 20, "C": 16,
         "precision": "fp32", "rebuild": False},
        {"name": "local_96k_bf16", "kind": "local", "system": "water", "n": 96000, "F": 64, "T": 2, "K": 20, "C": 16,
         "precision": "bf16", "rebuild": False},
        # a stretch of NVE on the device-resident loop, state in and out
        {"name": "md_water_6k_fp32", "kind": "md", "system": "water", "n": 6000, "F": 64, "T": 3, "K": 20,
         "precision": "fp32", "steps": 20, "dt": 0.5},
        # a batch of uneven replicas served together from submission to their results
        {"name": "serve_24_fp32", "kind": "serve", "replicas": 24, "lo": 64, "hi": 4000, "F": 64, "T": 3, "K": 20,
         "precision": "fp32", "steps": 8, "dt": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "call", "call", "call", "grad", "local", "md", "serve"])
    prec = rng.choice(["fp32", "bf16"])
    K = rng.choice([20, 20, 20, 16, 32])
    if kind == "serve":
        hi = _log_int(rng, 400, 6000)
        return {"kind": kind, "replicas": rng.randint(4, 24), "lo": 64, "hi": hi, "F": 64, "T": rng.choice([2, 3]), "K": 20,
                "precision": "fp32", "steps": rng.randint(4, 10), "dt": 0.5}
    if kind == "md":
        return {"kind": kind, "system": rng.choice(["water", "fcc"]), "n": _log_int(rng, 150, 20000),
                "F": rng.choice([64, 128]), "T": rng.choice([2, 3]), "K": K, "precision": "fp32",
                "steps": rng.randint(4, 20), "dt": 0.5}
    if kind == "local":
        return {"kind": kind, "system": rng.choice(["water", "fcc"]), "n": _log_int(rng, 150, 90000), "F": 64,
                "T": rng.choice([1, 2, 3]), "K": 20, "C": rng.choice([16, 32]), "precision": prec,
                "rebuild": rng.random() < 0.3}
    if kind == "grad":
        return {"kind": kind, "system": "mixture", "n": _log_int(rng, 1500, 90000), "F": 64, "T": 2, "K": K,
                "precision": prec}
    F = rng.choice([64, 128]) if prec == "bf16" else rng.choice([32, 64, 64, 128, 128, 256])
    system = rng.choice(["water", "fcc"])
    most = {32: 200000, 64: 250000, 128: 150000, 256: 20000}[F]
    if prec == "bf16" and F == 128 and system == "fcc":
        most = 700000
    return {"kind": kind, "system": system, "n": _log_int(rng, 150, most), "F": F, "T": rng.choice([2, 3, 3]), "K": K,
            "precision": prec, "rebuild": rng.random() < 0.3}


# ------------------------------------------------------------------------------ inputs
def _system(kind, n, seed):
    if kind == "water":
        return syn.water_box(max(1, n // 3), seed=seed)
    if kind == "mixture":
        chain = max(30, n // 300)
        return syn.mixture(n_chain=chain, n_water=(n - chain) // 3, seed=seed)
    side = (n / 4.0) ** (1.0 / 3.0)
    n1 = max(2, int(side))
    n2 = max(2, int(round(math.sqrt(n / 4.0 / n1))))
    n3 = max(2, int(round(n / 4.0 / (n1 * n2))))
    return syn.fcc(n1, n2, n3, jitter=0.05, seed=seed)


def _species(kind):
    return {"water": 2, "fcc": 1, "mixture": 4}[kind]


def _values(case, S, seed):
    """Weights with nonzero biases: a trained model has them."""
    if case["kind"] == "local":
        return syn.local_xavier_params(case["F"], case["K"], case["T"], S, case["C"], seed=seed, bias_scale=0.1)
    return syn.xavier_params(case["F"], case["K"], case["T"], S, seed=seed, bias_scale=0.1)


def _potential(case, S, seed):
    v = _values(case, S, seed)
    if case["kind"] == "local":
        blob = syn.local_params_blob(case["F"], case["K"], case["T"], S, case["C"], rc=RC, values=v)
        return eng.Potential(case["F"], K=case["K"], T=case["T"], n_species=S, rc=RC, precision=case["precision"],
                             params=blob, family="local", channels=case["C"])
    blob = syn.params_blob(case["F"], case["K"], case["T"], S, rc=RC, values=v)
    return eng.Potential(case["F"], K=case["K"], T=case["T"], n_species=S, rc=RC, precision=case["precision"], params=blob)


def _replicas(case, seed):
    """Replica systems of a serving session: sizes log-uniform, water and fcc in turn; the sizes
    belong to the case, the configurations and velocities to the seed."""
    sizes = syn.request_sizes(case["replicas"], case["lo"], case["hi"], seed=0)
    out = []
    for k, m in enumerate(sizes):
        sy = _system("water" if k % 2 == 0 else "fcc", int(m), seed + k)
        out.append((sy, syn.maxwell_boltzmann(sy.masses, 300.0, seed=seed + k)))
    return out


def prepare(case, seed):
    dev = DEV
    if case["kind"] == "serve":
        blob = syn.params_blob(case["F"], case["K"], case["T"], 2, rc=RC, values=_values(case, 2, seed))
        srv = eng.Server(case["F"], blob, K=case["K"], T=case["T"], n_species=2, rc=RC, precision=case["precision"],
                         max_replicas=case["replicas"], dt=case["dt"])
        return {"case": case, "srv": srv, "reps": _replicas(case, seed)}
    sy = _system(case["system"], case["n"], seed)
    pot = _potential(case, _species(case["system"]), seed)
    st = {"case": case, "sys": sy, "pot": pot, "cell": sy.cell}
    if case["kind"] == "md":
        st["vel"] = syn.maxwell_boltzmann(sy.masses, 300.0, seed=seed)
        return st
    st["z"] = torch.from_numpy(sy.species).to(dev)
    st["x"] = torch.from_numpy(sy.positions).to(dev)
    if case["kind"] == "grad":
        st["x"].requires_grad_(True)
    return st


# ------------------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        return _run_serve(state)
    pot = state["pot"]
    if kind == "md":
        sy = state["sys"]
        pot.md_set_state(sy.species, sy.masses, sy.positions, state["vel"], state["cell"], skin=1.0)
        ep, ek, _ = pot.md_run(case["steps"], case["dt"])
        x, v = pot.md_get_state()
        return {"epot": ep.astype(np.float32), "ekin": ek.astype(np.float32), "positions": x.astype(np.float32),
                "velocities": v.astype(np.float32)}
    keep = torch.float32 if case["precision"] == "fp32" else torch.bfloat16
    if kind == "grad":
        x = state["x"]
        x.grad = None
        e, w = eng.PaiNNEnergy.apply(x, state["z"], state["cell"], pot)
        e.backward()
        return {"energy": e.detach().to(keep), "virial": w.to(keep), "grad": x.grad.to(keep)}
    out = pot.compute(state["z"], state["x"], state["cell"], rebuild=case["rebuild"], energies=True)
    return {k: out[k].to(keep) for k in ("energy", "energies", "forces", "virial")}


def _run_serve(state):
    case, srv = state["case"], state["srv"]
    ids = [srv.submit(sy.species, sy.masses, sy.positions, v, sy.cell, nsteps=case["steps"]) for sy, v in state["reps"]]
    left = len(ids)
    while left:
        _, _, done = srv.step()
        left -= done
    got = [srv.poll(r) for r in ids]
    return {k: np.concatenate([g[k].reshape(-1) for g in got]).astype(np.float32)
            for k in ("epot", "ekin", "positions", "velocities", "virial")}


# ------------------------------------------------------------------------------ work
def work(case):
    """What one pass cannot do without: FLOPs of the contractions and elementwise terms of the model
    (forward and adjoint), bytes of the inputs, outputs and weights."""
    F, K, T = case["F"], case["K"], case["T"]
    per_edge, per_atom = 2 * T * (6 * K + 22) * F, 2 * T * 30 * F * F + F * F
    weights = 8 * T * (13 * F * F + 3 * F * K)
    if case["kind"] == "local":
        C = case["C"]
        layer = F * 2 * C + (F + 2 * C) * F
        mix = 4 * 2 * C * C
        per_edge = 2 * 2 * ((K + 4) * F + F * 2 * C + T * layer + (T - 1) * mix + F * F // 2)
        per_atom, weights = 0, 8 * ((K + 4) * F + 2 * F * C + T * layer + F * F // 2)
    edges = {"water": 51.5, "fcc": 35.0, "mixture": 51.5}
    if case["kind"] == "serve":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        atoms, n_e, evals, io = case["replicas"] * mean, 43.0, case["steps"] + 1, 28 + 8 + 24 + 48
    else:
        atoms, n_e = case["n"], edges[case["system"]]
        evals, io = (case["steps"] + 1, 28 + 8 + 24 + 48) if case["kind"] == "md" else (1, 28 + 24 + 8)
    return {"bytes": int(atoms * io + weights), "flops": int(evals * atoms * (per_atom + n_e * per_edge))}


# ------------------------------------------------------------------------------ 64-bit values
def _edges(x, H):
    """(i, j, r_j - r_i + image) of every directed pair within the cutoff, in 64 bits."""
    n, dev = x.shape[0], x.device
    inv = torch.linalg.inv(H)
    width = 1.0 / torch.linalg.norm(inv, dim=0)      # distance between opposite faces
    f = x @ inv
    f = f - torch.floor(f)
    reach = [int(math.floor(RC / w)) + 1 for w in width.tolist()]
    single = bool((width >= 2 * RC).all())
    images = [(0, 0, 0)] if single else [(a, b, c) for a in range(-reach[0], reach[0] + 1)
                                         for b in range(-reach[1], reach[1] + 1) for c in range(-reach[2], reach[2] + 1)]
    step = max(1, min(n, 40_000_000 // max(n, 1)))
    I, J, R = [], [], []
    for i0 in range(0, n, step):
        df = f[None] - f[i0:i0 + step, None]
        if single:
            df = df - torch.round(df)
        for im in images:
            shift = torch.tensor(im, dtype=torch.float64, device=dev)
            d = (df + shift) @ H
            ok = (d * d).sum(-1) < RC * RC
            if im == (0, 0, 0):
                k = torch.arange(ok.shape[0], device=dev)
                ok[k, k + i0] = False
            a, b = torch.nonzero(ok, as_tuple=True)
            I.append(a + i0)
            J.append(b)
            R.append(d[a, b])
    return torch.cat(I), torch.cat(J), torch.cat(R)


def _radial(r, K):
    d = torch.linalg.norm(r, dim=1)
    sig = RC / (K - 1)
    fc = 0.5 * (torch.cos(math.pi * d / RC) + 1)
    rbf = torch.exp(-(d[:, None] - sig * torch.arange(K, device=r.device, dtype=r.dtype)) ** 2 / (2 * sig * sig))
    return r / d[:, None], fc, rbf * fc[:, None]


def _painn(case, vals, S, z, i, j, r):
    F, K, T = case["F"], case["K"], case["T"]
    P = {k: torch.from_numpy(v).to(r.device) for k, v in syn.unpack_params(vals, F, K, T, S).items()}
    silu, n = torch.nn.functional.silu, z.shape[0]

    def layer(s, v, u, b, t):
        W1, b1, W2, b2, Wf, bf, U, V, A1, c1, A2, c2 = (P["%s_%d" % (k, t)] for k in (
            "W1", "b1", "W2", "b2", "Wf", "bf", "U", "V", "A1", "c1", "A2", "c2"))
        phi = silu(s @ W1.T + b1) @ W2.T + b2
        m = phi[j] * (b @ torch.cat([Wf, bf[:, None]], 1).T)
        s = s.index_add(0, i, m[:, :F])
        v = v.index_add(0, i, v[j] * m[:, None, F:2 * F] + u[:, :, None] * m[:, None, 2 * F:])
        Uv, Vv = v @ U.T, v @ V.T
        a = silu(torch.cat([s, torch.sqrt((Vv * Vv).sum(1) + 1e-8)], 1) @ A1.T + c1) @ A2.T + c2
        v = v + a[:, None, :F] * Uv
        return s + a[:, 2 * F:] + a[:, F:2 * F] * (Uv * Vv).sum(1), v

    u, fc, b = _radial(r, K)
    b = torch.cat([b, fc[:, None]], 1)
    s, v = P["emb"][z], torch.zeros(n, 3, F, dtype=r.dtype, device=r.device)
    for t in range(T):
        s, v = checkpoint(layer, s, v, u, b, t, use_reentrant=False)
    return silu(s @ P["R1"].T + P["d1"]) @ P["R2"] + P["d2"]


def _local(case, vals, S, z, i, j, r):
    F, K, L, C = case["F"], case["K"], case["T"], case["C"]
    P, off = {}, 0
    for name, shape in syn.local_param_shapes(F, K, L, S, C):
        m = int(np.prod(shape))
        P[name] = torch.from_numpy(vals[off:off + m].reshape(shape)).to(r.device)
        off += m
    silu, n = torch.nn.functional.silu, z.shape[0]
    u, fc, b = _radial(r, K)
    hot = torch.eye(S, dtype=r.dtype, device=r.device)
    x = silu(torch.cat([b, hot[z[i]], hot[z[j]]], 1) @ P["A0"] + P["c0"])
    w0 = x @ P["P0"]
    s, v = w0[:, :C], w0[:, None, C:] * u[:, :, None]

    def layer(x, s, v, u, fc, l):
        om = (x @ P["Q%d" % l]) * fc[:, None]
        zero = torch.zeros(n, 3, C, dtype=r.dtype, device=r.device)
        G = zero[:, 0].index_add(0, i, om[:, :C])[i]
        Gv = zero.index_add(0, i, om[:, None, C:] * u[:, :, None])[i]
        ts = torch.cat([s * G, (v * Gv).sum(1)], 1)
        if l < L:
            v = torch.cat([s[:, None] * Gv, v * G[:, None]], 2) @ P["Gv%d" % l]
            s = ts @ P["Gs%d" % l]
        return silu(torch.cat([x, ts], 1) @ P["M%d" % l] + P["m%d" % l]), s, v

    for l in range(1, L + 1):
        x, s, v = checkpoint(layer, x, s, v, u, fc, l, use_reentrant=False)
    y = fc * (silu(x @ P["R1"] + P["d1"]) @ P["R2"] + P["d2"])
    return torch.zeros(n, dtype=r.dtype, device=r.device).index_add(0, i, y)


def _evaluate(case, vals, S, z, x, H):
    """Per-atom energies, forces and virial by automatic differentiation, in 64 bits."""
    i, j, r = _edges(x, H)
    r.requires_grad_(True)
    e = (_local if case["kind"] == "local" else _painn)(case, vals, S, z, i, j, r)
    (g,) = torch.autograd.grad(e.sum(), r)
    f = torch.zeros_like(x).index_add(0, i, g).index_add(0, j, -g)
    return e.detach(), f, -(r.detach().T @ g)


def _nve(case, vals, S, sy, vel):
    """Velocity Verlet in 64 bits: (epot, ekin per step, positions, velocities, last virial)."""
    dev = DEV
    z, m = torch.from_numpy(sy.species).to(dev).long(), torch.from_numpy(sy.masses).to(dev)[:, None]
    x, v, H = (torch.from_numpy(a).to(dev) for a in (sy.positions.copy(), vel.copy(), sy.cell))
    dt, ep, ek = case["dt"], [], []
    for k in range(case["steps"] + 1):
        if k:
            v = v + 0.5 * dt * ACC * f / m
            x = x + dt * v
        e, f, w = _evaluate(case, vals, S, z, x, H)
        if k:
            v = v + 0.5 * dt * ACC * f / m
        ep.append(e.sum())
        ek.append((0.5 * m * v * v).sum() / ACC)
    return torch.stack(ep), torch.stack(ek), x, v, w


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        vals, parts = _values(case, 2, seed), []
        if case["replicas"] * case["hi"] * case["steps"] > 1_200_000:
            return None
        for sy, v in _replicas(case, seed):
            parts.append([p.reshape(-1) for p in _nve(case, vals, 2, sy, v)])
        return dict(zip(("epot", "ekin", "positions", "velocities", "virial"), (torch.cat(p) for p in zip(*parts))))
    S = _species(case["system"])
    per_edge = case["F"] * 3 * 8 if kind != "local" else (case["F"] * 4 + case["C"] * 20) * 8
    cost = case["n"] * {"water": 52, "fcc": 36, "mixture": 52}[case["system"]] * per_edge
    vals = _values(case, S, seed)
    sy = _system(case["system"], case["n"], seed)
    if kind == "md":
        if cost * case["steps"] > 2e11:
            return None
        ep, ek, x, v, _ = _nve(case, vals, S, sy, syn.maxwell_boltzmann(sy.masses, 300.0, seed=seed))
        return {"epot": ep, "ekin": ek, "positions": x, "velocities": v}
    if cost > (2.5e10 if kind == "local" else 1.2e10):
        return None
    dev = DEV
    e, f, w = _evaluate(case, vals, S, torch.from_numpy(sy.species).to(dev).long(),
                        torch.from_numpy(sy.positions).to(dev), torch.from_numpy(sy.cell).to(dev))
    # totals of the BF16 path: what is left when the errors of all atoms, of either sign, cancel; it is
    # no measure of the path's precision, the per-atom energies and forces are
    whole = case["precision"] == "fp32"
    out = {"energy": e.sum() if whole else None, "virial": w if whole else None}
    if kind == "grad":
        out["grad"] = -f
    else:
        out["forces"], out["energies"] = f, e
        out["energy"] = e.sum().reshape(1) if whole else None
    return out
