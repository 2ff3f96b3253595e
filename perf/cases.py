"""Workloads by which the speed of the library is judged, each through its public entry points.

The library serves programs that hand it the bodies of a regularised region and read the
integrated state back, so most cases here are one pass of such a loop: the state goes in, one
GBS step (or one force evaluation, one tree) is taken, the state comes out. The others are the
batched systems, the differentiable fixed-step run and the rebuild experiment of Sec. 3.5.

Every pass starts from the same state with a given fictitious step, so that it does the same
work each time it is called. The tolerance is 1e-11 and the steps are short enough for the
extrapolation error to lie at its rounding floor (a few 1e-13): a step is then accepted at the
first attempt whatever the last bits of the arithmetic are. The error estimate itself, which is
rounding noise at that level, is not among the outputs, nor is the next step derived from it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2001_03180_gb300 import mstar as M
from paper_2001_03180_gb300 import workloads as W

ETA = 1e-11
T_END = 1e6      # far beyond any pass: no step is clamped to an end time
FLOPS_PAIR = 33  # algorithmic FP64 flops of one unordered pair interaction


def listed():
    return [
        # A regularised binary on its own: the smallest call, all launches and latency.
        {"name": "step_kepler2", "kind": "step", "model": "kepler", "n": 2, "k_fix": 8},
        # A small star cluster (the repository's Plummer 64 configuration).
        {"name": "step_plummer64", "kind": "step", "model": "plummer", "n": 64, "k_fix": 8},
        # A region of a few hundred stars around an SMBH binary, a ragged size.
        {"name": "step_smbh601", "kind": "step", "model": "smbh_binary", "n": 601, "k_fix": 8},
        # The Plummer 2048 + SMBH binary configuration.
        {"name": "step_smbh2050", "kind": "step", "model": "smbh_binary", "n": 2050, "k_fix": 8},
        # The headline configuration: 10^4 stars and two SMBHs, one accepted GBS step.
        {"name": "step_smbh10002", "kind": "step", "model": "two_smbh", "n": 10002, "k_fix": 8},
        # Forces on a new state (tree, edge vectors, pair loop) for a program with its own
        # integrator; an odd size.
        {"name": "forces5003", "kind": "forces", "model": "plummer", "n": 5003},
        # The allocation-free pair loop on device arrays, inside a host code's own loop.
        {"name": "forces_noalloc2047", "kind": "noalloc", "n": 2047},
        # Many independent systems at once: triples and clusters of 3 to 199 bodies.
        {"name": "batch_mixed1024", "kind": "batch", "systems": 1024, "n_max": 199, "triples": False},
        # A population of hierarchical triples: the smallest systems of a batch.
        {"name": "batch_triples2048", "kind": "batch", "systems": 2048, "n_max": 3, "triples": True},
        # Forward run and gradients of a differentiable fixed-step run (Plummer 256).
        {"name": "adjoint256", "kind": "adjoint", "n": 256, "nsteps": 20, "every": 10},
        # The rebuild test of Sec. 3.5 on one Hernquist cluster: both coordinate systems, all
        # four deconstruction rules.
        {"name": "rebuild379", "kind": "rebuild", "n": 379, "cycles": 1000, "topo_every": 1000},
        # The divide-and-conquer tree of Sec. 3.3 at the headline size.
        {"name": "tree_dc10002", "kind": "tree", "n": 10002},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "forces", "noalloc", "batch", "adjoint", "rebuild", "tree"])
    if kind == "step":
        n = _log_int(rng, 2, 10001)
        model = "kepler" if n == 2 else ("plummer" if n < 16 else rng.choice(["plummer", "smbh_binary"]))
        return {"kind": kind, "model": model, "n": n, "k_fix": rng.choice([6, 7, 8])}
    if kind == "forces":
        return {"kind": kind, "model": rng.choice(["plummer", "smbh_binary"]), "n": _log_int(rng, 16, 5002)}
    if kind == "noalloc":
        return {"kind": kind, "n": _log_int(rng, 2, 2046)}
    if kind == "batch":
        triples = rng.random() < 0.3
        return {"kind": kind, "systems": _log_int(rng, 32, 2047 if triples else 1023),
                "n_max": 3 if triples else _log_int(rng, 8, 199), "triples": triples}
    if kind == "adjoint":
        return {"kind": kind, "n": _log_int(rng, 16, 255), "nsteps": rng.randint(4, 19), "every": rng.randint(2, 10)}
    if kind == "rebuild":
        return {"kind": kind, "n": _log_int(rng, 32, 378), "cycles": rng.randint(100, 999),
                "topo_every": rng.choice([100, 250, 1000])}
    return {"kind": kind, "n": _log_int(rng, 64, 10001)}


# ---------------------------------------------------------------------------- inputs

def _system(case, seed):
    n, model = case["n"], case.get("model", "plummer")
    if model == "kepler":
        return W.kepler_binary(seed, m1=0.6, m2=0.4, true_anomaly=2.0 + (seed % 97) / 97.0)
    if model == "smbh_binary":
        return W.plummer_smbh_binary(n - 2, seed)
    if model == "two_smbh":
        return W.plummer_two_smbh(n - 2, seed)
    return W.plummer(n, seed)


def _fict_step(n):
    """Fictitious step well inside the tolerance for the systems of _system."""
    return 2e-3 if n <= 256 else 3e-4


def _batch_systems(case, seed):
    if case["triples"]:
        st = W.Stream(seed, 23)
        out = []
        for _ in range(case["systems"]):
            e, a, inc = st.uniform(3)
            out.append(W.hierarchical_triple(1.0, 1.0, 0.1, 1.0, 0.9 * e, 10.0 + 40.0 * a, 0.0,
                                             math.radians(40.0 + 100.0 * inc), st))
        return out
    # the sizes of W.batched_systems' mix, the same for every seed: a triple, then a cluster with a
    # central mass of a tenth of its stars', the clusters spread evenly over the logarithm of n
    half = case["systems"] // 2
    triples = _batch_systems({"systems": case["systems"] - half, "triples": True}, seed)
    out = []
    for i in range(case["systems"]):
        if i % 2 == 0:
            out.append(triples[i // 2])
            continue
        n = max(3, int(round(3.0 * (case["n_max"] / 3.0) ** ((i // 2 + 0.5) / half))))
        m, r, v = W.plummer(n - 1, seed * 100003 + i)
        m = np.concatenate([m, [0.1 * m.sum()]])
        out.append((m, np.concatenate([r, np.zeros((1, 3))]), np.concatenate([v, np.zeros((1, 3))])))
    return out


def _batch_H(systems):
    return np.array([2e-2 if len(s[0]) == 3 else 1e-3 for s in systems])


def _loss_weights(n, seed):
    st = W.Stream(seed, 5)
    return st.uniform(3 * n).reshape(n, 3) - 0.5, st.uniform(3 * n).reshape(n, 3) - 0.5, 0.7


def _rebuild_jobs(case, seed):
    m, r, v, _ = W.hernquist(case["n"], seed)
    jobs = [(c, d) for c in (0, 1) for d in (0, 1, 2, 3)]
    return (m, r, v), [j[0] for j in jobs], [j[1] for j in jobs]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "forces", "tree"):
        m, r, v = _system(case, seed)
        params = {"eta_gbs": ETA}
        if "k_fix" in case:
            params["k_fix"] = case["k_fix"]
        if kind == "tree":
            params["mst_method"] = 1
        return {"kind": kind, "g": M.Integrator(m, r, v, **params), "r": r, "v": v, "H": _fict_step(case["n"])}
    if kind == "noalloc":
        m, r, _ = W.plummer(case["n"], seed)
        dev = torch.device("cuda")
        return {"kind": kind, "n": case["n"], "m": torch.from_numpy(m).to(dev), "r": torch.from_numpy(r).to(dev),
                "a": torch.empty(case["n"], 3, dtype=torch.float64, device=dev),
                "U": torch.empty(1, dtype=torch.float64, device=dev)}
    if kind == "batch":
        systems = _batch_systems(case, seed)
        return {"kind": kind, "b": M.Batch(systems, eta_gbs=ETA), "H": _batch_H(systems)}
    if kind == "adjoint":
        m, r, v = W.plummer(case["n"], seed)
        wr, wv, we = _loss_weights(case["n"], seed)
        cuda = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        return {"kind": kind, "m": cuda(m), "r": cuda(r), "v": cuda(v), "wr": cuda(wr), "wv": cuda(wv), "we": we,
                "H": _fict_step(case["n"]), "nsteps": case["nsteps"], "every": case["every"]}
    if kind == "rebuild":
        system, coords, decon = _rebuild_jobs(case, seed)
        return {"kind": kind, "systems": [system] * len(coords), "coords": coords, "decon": decon,
                "cycles": case["cycles"], "topo_every": case["topo_every"], "sample_at": [0, case["cycles"]]}
    raise ValueError(kind)


# ---------------------------------------------------------------------------- one pass

def run(state):
    kind = state["kind"]
    if kind == "step":
        g = state["g"]
        g.set_state(0.0, state["r"], state["v"])
        g.set_H(state["H"])
        _, stats = g.step(T_END, max_steps=1)
        out = g.state()
        return {"t": out["t"], "r": out["r"], "v": out["v"], "accepted": stats["accepted"],
                "rejected": stats["rejected"], "force_evals": stats["force_evals"]}
    if kind == "forces":
        g = state["g"]
        g.set_state(0.0, state["r"], state["v"])
        a, U = g.accelerations()
        return {"a": a, "U": U}
    if kind == "tree":
        g = state["g"]
        g.set_state(0.0, state["r"], state["v"])
        root, parent, level, _ = g.mst(with_order=False)
        return {"root": root, "parent": parent, "level": level}
    if kind == "noalloc":
        rc = M.mstar_accelerations_noalloc(state["n"], state["m"], state["r"], 1.0, state["a"], state["U"],
                                           torch.cuda.current_stream().cuda_stream)
        if rc != M.MSTAR_OK:
            raise M.MstarError(rc, "mstar_accelerations_noalloc")
        return {"a": state["a"], "U": state["U"]}
    if kind == "batch":
        b = state["b"]
        b.set_H(state["H"])
        b.step(T_END, 1)
        out = b.state()
        return {"t": out["t"], "r": np.concatenate(out["r"]), "v": np.concatenate(out["v"]), "status": out["status"]}
    if kind == "adjoint":
        m, r, v = (state[k].clone().requires_grad_(True) for k in ("m", "r", "v"))
        rf, vf, E = M.fixed_run(m, r, v, H=state["H"], nsteps=state["nsteps"], checkpoint_every=state["every"])
        loss = (state["wr"] * rf).sum() + (state["wv"] * vf).sum() + state["we"] * E
        loss.backward()
        return {"r": rf.detach(), "v": vf.detach(), "E": E.detach(), "dm": m.grad, "dr": r.grad, "dv": v.grad}
    out = M.mstar_rebuild_test(state["systems"], state["coords"], state["decon"], state["cycles"],
                               state["topo_every"], state["sample_at"])
    return {k: out[k] for k in ("E", "r", "v", "topo_changes", "mean_level")}


# ---------------------------------------------------------------------------- what a pass needs

def _evals(k_fix):
    """Force evaluations of one attempt: the divisions' 2 + 4 + ... + 2 k_fix and the step start."""
    return k_fix * (k_fix + 1) + 1


def work(case):
    kind = case["kind"]
    if kind == "batch":
        # mean sizes: triples alternate with clusters whose size is uniform in its logarithm
        if case["triples"]:
            bodies, pairs = 3.0, 3.0
        else:
            span = math.log(case["n_max"] / 3.0) if case["n_max"] > 3 else 1e-9
            mean = (case["n_max"] - 3.0) / span
            mean2 = (case["n_max"] ** 2 - 9.0) / (2.0 * span)
            bodies, pairs = 0.5 * (3.0 + mean), 0.5 * (3.0 + 0.5 * (mean2 - mean))
        return {"bytes": case["systems"] * bodies * 8 * 13, "flops": case["systems"] * pairs * FLOPS_PAIR * _evals(8)}
    n = case["n"]
    pairs = 0.5 * n * (n - 1)
    if kind == "step":
        return {"bytes": 8.0 * 13 * n, "flops": pairs * FLOPS_PAIR * _evals(case["k_fix"])}
    if kind == "forces":
        return {"bytes": 8.0 * 10 * n, "flops": pairs * FLOPS_PAIR}
    if kind == "noalloc":
        return {"bytes": 8.0 * 7 * n, "flops": pairs * FLOPS_PAIR}
    if kind == "adjoint":
        # the forward's evaluations and one vector-Jacobian product (about 70 flops a pair) for each
        return {"bytes": 8.0 * 27 * n, "flops": case["nsteps"] * pairs * _evals(8) * (FLOPS_PAIR + 70)}
    if kind == "rebuild":
        # building and taking apart two 3-vectors per body and cycle, for eight jobs
        return {"bytes": 8 * 8.0 * 13 * n, "flops": 8 * case["cycles"] * 12.0 * n}
    return {"bytes": 8.0 * 6 * n + 8.0 * n, "flops": pairs * 8}


# ---------------------------------------------------------------------------- values in plain torch

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _forces(m, r, live):
    """Accelerations and the force function of S systems of n bodies (m [S, n], r [S, n, 3], G = 1)."""
    S, n = m.shape
    a = torch.empty_like(r)
    U = torch.zeros(S, dtype=r.dtype, device=r.device)
    rows = max(1, min(n, (1 << 26) // max(1, S * n)))
    idx = torch.arange(n, device=r.device)
    for i0 in range(0, n, rows):
        i1 = min(n, i0 + rows)
        d = r[:, None, :, :] - r[:, i0:i1, None, :]
        r2 = (d * d).sum(-1)
        keep = live[:, None, :] & live[:, i0:i1, None] & (idx[None, i0:i1, None] != idx[None, None, :])
        inv = torch.where(keep, torch.where(keep, r2, torch.ones_like(r2)).rsqrt(), torch.zeros_like(r2))
        w = m[:, None, :] * inv
        U = U + 0.5 * (m[:, i0:i1] * w.sum(-1)).sum(-1)
        a[:, i0:i1] = ((w * inv * inv)[..., None] * d).sum(2)
    return a, U


def _kinetic(m, v):
    return 0.5 * (m * (v * v).sum(-1)).sum(-1)


def _gbs(m, r, v, t, B, H, k_fix, forces):
    """One GBS step of the LogH leapfrog in Cartesian coordinates (equal to the step in edge
    vectors in real arithmetic): the k_fix divisions and their extrapolation to step length 0."""
    x = [1.0 / (2.0 * k) ** 2 for k in range(1, k_fix + 1)]
    col = lambda f: f[:, None, None]  # noqa: E731
    out = None
    for k in range(1, k_fix + 1):
        c = 1.0
        for j in range(k_fix):
            if j != k - 1:
                c *= x[j] / (x[j] - x[k - 1])
        nk = 2 * k
        delta = H / nk
        f = 0.5 * delta / (_kinetic(m, v) + B)
        rk, vk, tk = r + col(f) * v, v, t + f
        for tau in range(1, nk + 1):
            a, U = forces(m, rk)
            vk = vk + col(delta / U) * a
            f = (0.5 if tau == nk else 1.0) * delta / (_kinetic(m, vk) + B)
            rk = rk + col(f) * vk
            tk = tk + f
        part = (c * rk, c * vk, c * tk)
        out = part if out is None else tuple(p + q for p, q in zip(out, part))
    return out


def _com(m, x):
    return x - (m[:, :, None] * x).sum(1, keepdim=True) / m.sum(1)[:, None, None]


def _step_exact(systems, H, k_fix):
    dev = _dev()
    n = max(len(s[0]) for s in systems)
    S = len(systems)
    m = torch.zeros(S, n, dtype=torch.float64)
    r = torch.zeros(S, n, 3, dtype=torch.float64)
    v = torch.zeros(S, n, 3, dtype=torch.float64)
    live = torch.zeros(S, n, dtype=torch.bool)
    for s, (ms, rs, vs) in enumerate(systems):
        k = len(ms)
        m[s, :k], r[s, :k], v[s, :k], live[s, :k] = map(torch.from_numpy, (ms, rs, vs, np.ones(k, bool)))
    m, r, v, live = m.to(dev), r.to(dev), v.to(dev), live.to(dev)
    r, v = _com(m, r), _com(m, v)
    forces = lambda mm, rr: _forces(mm, rr, live)  # noqa: E731
    B = forces(m, r)[1] - _kinetic(m, v)
    t = torch.zeros(S, dtype=torch.float64, device=dev)
    r, v, t = _gbs(m, r, v, t, B, torch.as_tensor(H, dtype=torch.float64, device=dev), k_fix, forces)
    r, v = _com(m, r), _com(m, v)
    return t.cpu().numpy(), r[live].cpu().numpy(), v[live].cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        t, r, v = _step_exact([_system(case, seed)], [_fict_step(case["n"])], case["k_fix"])
        return {"t": float(t[0]), "r": r, "v": v, "accepted": None, "rejected": None, "force_evals": None}
    if kind == "batch":
        systems = _batch_systems(case, seed)
        t, r, v = _step_exact(systems, _batch_H(systems), 8)
        return {"t": t, "r": r, "v": v, "status": None}
    if kind in ("forces", "noalloc"):
        m, r, _ = _system(case, seed)
        m, r = (torch.from_numpy(x).to(_dev())[None] for x in (m, r))
        a, U = _forces(m, r, torch.ones_like(m, dtype=torch.bool))
        return {"a": a[0].cpu().numpy(), "U": float(U[0]) if kind == "forces" else U.cpu().numpy()}
    if kind == "adjoint":
        dev, n = _dev(), case["n"]
        m, r, v = (torch.from_numpy(x).to(dev).requires_grad_(True) for x in W.plummer(n, seed))
        wr, wv, we = _loss_weights(n, seed)
        off = ~torch.eye(n, dtype=torch.bool, device=dev)

        def forces(mm, rr):
            d = rr[:, None, :, :] - rr[:, :, None, :]
            r2 = (d * d).sum(-1)
            inv = torch.where(off, torch.where(off, r2, torch.ones_like(r2)).rsqrt(), torch.zeros_like(r2))
            w = mm[:, None, :] * inv
            return ((w * inv * inv)[..., None] * d).sum(2), 0.5 * (mm * w.sum(-1)).sum(-1)

        mm = m[None]
        x, u = _com(mm, r[None]), _com(mm, v[None])
        B = forces(mm, x)[1] - _kinetic(mm, u)
        t = torch.zeros(1, dtype=torch.float64, device=dev)
        H = torch.full((1,), _fict_step(n), dtype=torch.float64, device=dev)
        for _ in range(case["nsteps"]):
            x, u, t = _gbs(mm, x, u, t, B, H, 8, forces)
        E = (_kinetic(mm, u) - forces(mm, x)[1])[0]
        loss = (torch.from_numpy(wr).to(dev) * x[0]).sum() + (torch.from_numpy(wv).to(dev) * u[0]).sum() + we * E
        loss.backward()
        return {"r": x[0].detach(), "v": u[0].detach(), "E": E.detach(), "dm": m.grad, "dr": r.grad, "dv": v.grad}
    if kind == "rebuild":
        # building the relative coordinates and taking them apart is the identity, up to the
        # centre-of-mass shift of rules 0 and 3; the energy does not change
        (m, r, v), coords, decon = _rebuild_jobs(case, seed)
        d = r[:, None, :] - r[None, :, :]
        with np.errstate(divide="ignore"):
            inv = 1.0 / np.sqrt((d * d).sum(-1))
        np.fill_diagonal(inv, 0.0)
        E = 0.5 * float((m * (v * v).sum(1)).sum()) - 0.5 * float((m[:, None] * m[None, :] * inv).sum())
        c = lambda x, k: x - (m[:, None] * x).sum(0) / m.sum() if k in (0, 3) else x  # noqa: E731
        return {"E": np.full((len(coords), 2), E), "r": np.stack([c(r, k) for k in decon]),
                "v": np.stack([c(v, k) for k in decon]), "topo_changes": None, "mean_level": None}
    return None
