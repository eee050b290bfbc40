"""Timed cases of the framework: what its users have it compute, through the package's own entry points.

A case is a dict of plain values.  Its "call" says which entry point it stands for:

  solve     init_uniform, evolve, observables: one adiabatic run of one 3-SAT instance
  schedule  the same over a caller's sin^2 sweep (evolve_schedule)
  order4    the same in fourth-order steps (evolve_order4)
  resume    a piece of a longer run (evolve_range), as between two checkpoints, then the observables
  observe   the observables of a state in hand
  spectrum  the lowest levels of H(s) (lowest_eigenvalues)
  serve     a mix of requests submitted to a running server at once, all results collected

Instances are planted 3-SAT: clauses drawn at random, those that the planted assignment falsifies dropped.
"""

import math
import time

import numpy as np
import torch

import paper_1103_1399_gb300 as q

# Clause counts of this repository's planted unique-solution instances lie between about 4 n and 15 n.
DT = 0.05  # Strang step of the small and mid-size configurations


def listed():
    return [
        # The six-variable worked example: the smallest run in use, all latency.
        {"name": "solve 6", "call": "solve", "n": 6, "m": 26, "T": 8.0, "steps": 80},
        # The 12-qubit configuration: one state in one SM's shared memory, 400 steps.
        {"name": "solve 12", "call": "solve", "n": 12, "m": 72, "T": 20.0, "steps": 400},
        # Middle of the served sizes, just above what one SM holds.
        {"name": "solve 16", "call": "solve", "n": 16, "m": 96, "T": 20.0, "steps": 400},
        # A non-linear sweep of a ratio-4.2 instance run as one launch graph.
        {"name": "sweep 19 graph", "call": "schedule", "n": 19, "m": 80, "T": 10.0, "steps": 200, "graph": True},
        # The 20-qubit configuration.
        {"name": "solve 20", "call": "solve", "n": 20, "m": 100, "T": 10.0, "steps": 200},
        # An odd size above the served range; the state (64 MiB) still fits in L2.
        {"name": "solve 23", "call": "solve", "n": 23, "m": 140, "T": 2.0, "steps": 40},
        # Fourth-order steps on a state beyond L2.
        {"name": "order4 26", "call": "order4", "n": 26, "m": 230, "T": 0.5, "steps": 5},
        # The headline configuration: eight of its 400 steps, from the middle of the sweep, and the observables.
        {"name": "resume 30", "call": "resume", "n": 30, "m": 371, "T": 40.0, "steps": 400, "k0": 196, "k1": 204},
        # The tensor-core precision variant (BF16 in three parts) of the configuration at 28 qubits.
        {"name": "tensor cores 28", "call": "solve", "n": 28, "m": 419, "T": 0.4, "steps": 4, "variant": 1},
        # The observables alone, as between the pieces of a run.
        {"name": "observe 29", "call": "observe", "n": 29, "m": 300},
        # One point of a gap scan at 20 qubits.
        {"name": "spectrum 20", "call": "spectrum", "n": 20, "m": 100, "s": 0.5, "levels": 2, "iters": 120},
        # The serving mix (n in 10..22, T in 5..80): 96 requests arriving at once.
        {"name": "serve 96", "call": "serve", "requests": 96, "n_lo": 10, "n_hi": 22, "t_lo": 5.0, "t_hi": 80.0},
    ]


def draw(rng):
    """One case of the ranges above; no drawn case costs more than the eight 30-qubit steps."""
    call = rng.choice(["solve", "solve", "solve", "solve", "schedule", "order4", "resume", "observe", "spectrum", "serve"])
    if call == "serve":
        lo = rng.randint(10, 16)
        t_lo = round(rng.uniform(5.0, 20.0), 2)
        return {"call": call, "requests": int(2 ** rng.uniform(2.0, 6.5)), "n_lo": lo, "n_hi": rng.randint(lo + 1, 22),
                "t_lo": t_lo, "t_hi": round(rng.uniform(t_lo, 80.0), 2)}
    if call == "spectrum":
        n = rng.randint(12, 24)
        return {"call": call, "n": n, "m": _clauses(rng, n), "s": round(rng.uniform(0.2, 0.9), 3), "levels": rng.randint(1, 2),
                "iters": rng.randint(100, 160)}
    if call == "observe":
        n = rng.randint(8, 29)
        return {"call": call, "n": n, "m": _clauses(rng, n)}
    n = rng.randint(5, 28)
    # steps spread over their logarithm, up to 400 and to a bounded amount of work
    most = max(3, min(400, (1 << 31) // (1 << n)))
    steps = int(2 ** rng.uniform(math.log2(3), math.log2(most + 0.5))) if most > 3 else 3
    case = {"call": call, "n": n, "m": _clauses(rng, n), "T": round(steps * rng.choice([0.05, 0.1]), 4), "steps": steps}
    if call == "resume":
        case["k0"] = rng.randint(0, steps - 2)
        case["k1"] = rng.randint(case["k0"] + 1, steps)
    if call == "order4":
        case["steps"] = max(1, steps // 3)
        case["T"] = round(case["steps"] * 0.1, 4)
    if call == "solve" and n >= 15:
        case["variant"] = rng.choice([-1, -1, -1, 0, 1, 2])
    if n >= 15 and rng.random() < 0.25:
        case["graph"] = True
    return case


def _clauses(rng, n):
    return int(n * rng.uniform(4.2, 13.0))


# ------------------------------------------------------------------ inputs ----
def _planted(n, m, rng):
    """m clauses of three distinct variables with random signs, none falsified by the planted assignment."""
    x = rng.integers(0, 2, size=n)
    out = []
    while len(out) < m:
        size = 2 * (m - len(out)) + 16
        vs = np.argsort(rng.random((size, n)), axis=1)[:, :3]
        sg = rng.integers(0, 2, size=(size, 3))
        good = (x[vs] == sg).any(axis=1)
        lits = np.where(sg == 1, vs + 1, -(vs + 1))[good]
        out.extend(lits[: m - len(out)].tolist())
    return out


def _requests(case, seed):
    rng = np.random.default_rng([seed, 7])
    reqs = []
    for _ in range(case["requests"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        T = float(rng.uniform(case["t_lo"], case["t_hi"]))
        reqs.append((n, _planted(n, int(n * rng.uniform(4.2, 8.0)), rng), T, max(1, round(T / DT))))
    return reqs


def _sweep(case):
    K = case["steps"]
    return np.sin(0.5 * np.pi * (np.arange(K) + 0.5) / K) ** 2


def _mid_run_state(n, seed):
    """A normalised product of n one-qubit states, each still close to the uniform start: the spread of
    magnitudes and phases of a run's middle."""
    rng = np.random.default_rng([seed, 3])
    a, phi = rng.uniform(0.5, 1.05, size=n), rng.uniform(-math.pi, math.pi, size=n)
    parts = [np.ones(1, dtype=np.complex128), np.ones(1, dtype=np.complex128)]
    for i in range(n):
        one = np.array([math.cos(a[i]), math.sin(a[i]) * complex(math.cos(phi[i]), math.sin(phi[i]))])
        k = 0 if i < n // 2 else 1
        parts[k] = (one[:, None] * parts[k][None, :]).reshape(-1)
    lo, hi = (torch.from_numpy(p.astype(np.complex64)).to(_device()) for p in parts)
    return (hi[:, None] * lo[None, :]).reshape(-1)


def prepare(case, seed):
    if case["call"] == "serve":
        # The running server and the requests' instances.
        return {"case": case, "server": q.Server(hbm_budget_bytes=4 << 30, max_slots=256), "requests": _requests(case, seed)}
    n = case["n"]
    inst = q.Instance(n, _planted(n, case["m"], np.random.default_rng([seed, n])))
    state = {"case": case, "inst": inst}
    if case["call"] == "spectrum":
        return state
    if case.get("variant", -1) >= 0:
        inst.set_variant(case["variant"])
    if case.get("graph"):
        inst.set_launch_mode(q.LAUNCH_GRAPH)
    if case["call"] == "observe":
        # Observables follow an evolution on the same handle.
        psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
        inst.init_uniform(psi)
        inst.evolve(psi, 0.1, 1)
        del psi
        state["psi"] = _mid_run_state(n, seed)
    elif case["call"] == "resume":
        state["start"] = _mid_run_state(n, seed)
        state["psi"] = torch.empty_like(state["start"])
    else:
        state["psi"] = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    if case["call"] == "schedule":
        state["s"] = _sweep(case).tolist()
    return state


# --------------------------------------------------------------------- run ----
def _serve(server, requests):
    tickets = [server.submit(n, clauses, T, K) for n, clauses, T, K in requests]
    done = {}
    while len(done) < len(tickets):
        for t in tickets:
            if t not in done:
                r = server.poll(t)
                if r is None:
                    break
                done[t] = r
        else:
            break
        time.sleep(0.0005)
    rows = [done[t] for t in tickets]
    # (numbers of complex64 states, hence of 32-bit accuracy)
    out = {k: np.array([r[k] for r in rows], dtype=np.float32) for k in ("success_prob", "energy", "norm", "expect_hb")}
    out["ground_count"] = np.array([r["ground_count"] for r in rows], dtype=np.int64)
    out["status"] = np.array([r["status"] for r in rows], dtype=np.int64)
    return out


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "serve":
        return _serve(state["server"], state["requests"])
    inst = state["inst"]
    if call == "spectrum":
        levels, iters = inst.lowest_eigenvalues(case["s"], k=case["levels"], max_iter=case["iters"])
        return {"levels": levels, "iters": iters}
    psi = state["psi"]
    if call == "observe":
        return inst.observables(psi)
    if call == "resume":
        # From the checkpointed state, which stays as it is.
        psi.copy_(state["start"])
        inst.evolve_range(psi, case["T"], case["steps"], case["k0"], case["k1"])
    else:
        inst.init_uniform(psi)
        if call == "schedule":
            inst.evolve_schedule(psi, case["T"] / case["steps"], state["s"])
        elif call == "order4":
            inst.evolve_order4(psi, case["T"], case["steps"])
        else:
            inst.evolve(psi, case["T"], case["steps"])
    return {"psi": psi, "observables": inst.observables(psi)}


# -------------------------------------------------------------------- work ----
def _sub_steps(case):
    if case["call"] == "resume":
        return case["k1"] - case["k0"]
    return case["steps"] * (3 if case["call"] == "order4" else 1)


def work(case):
    """Each input read and each output written once; per step and amplitude one complex phase multiply (6 operations)
    and one real rotation per qubit and component (4 operations per qubit)."""
    if case["call"] == "serve":
        sizes = [(n, 4.2 * n, 0.5 * (case["t_lo"] + case["t_hi"]) / DT) for n in range(case["n_lo"], case["n_hi"] + 1)]
        share = case["requests"] / len(sizes)
        flops = sum(share * K * 2.0**n * (4 * n + 6) for n, m, K in sizes)
        return {"bytes": sum(share * (12 * m + 48) for n, m, K in sizes), "flops": flops}
    n, N = case["n"], float(2 ** case["n"])
    if case["call"] == "spectrum":
        # n additions, the diagonal and three vector updates per amplitude and iteration; the clauses in, the levels out
        return {"bytes": 12.0 * case["m"] + 8 * case["levels"], "flops": case["iters"] * N * (n + 12)}
    if case["call"] == "observe":
        return {"bytes": 8 * N + 12 * case["m"], "flops": N * (2 * n + 8)}
    state_bytes = (16 if case["call"] == "resume" else 8) * N
    return {"bytes": state_bytes + 12 * case["m"], "flops": _sub_steps(case) * N * (4 * n + 6) + N * (2 * n + 8)}


# ------------------------------------------------------------------- exact ----
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _energies(n, clauses):
    """Violated-clause count of every index, int16."""
    dev = _device()
    out = torch.zeros(1 << n, dtype=torch.int16, device=dev)
    part = 1 << min(n, 24)
    for i in range(0, 1 << n, part):
        x = torch.arange(i, i + part, dtype=torch.int32, device=dev)
        for c in clauses:
            mask = sum(1 << (abs(l) - 1) for l in c)
            viol = sum(1 << (abs(l) - 1) for l in c if l < 0)
            out[i : i + part] += (x & mask) == viol
    return out


def _phase(psi, E, angle):
    """psi <- exp(-i angle E) psi, in pieces."""
    tab = torch.arange(int(E.max()) + 1, dtype=torch.float64, device=psi.device) * -angle
    tab = torch.complex(torch.cos(tab), torch.sin(tab))
    part = 1 << 26
    for i in range(0, psi.numel(), part):
        psi[i : i + part] *= tab[E[i : i + part].long()]


def _mix(psi, n, theta):
    """psi <- exp(-i theta sum_i (1 - X_i)/2) psi, one qubit at a time."""
    c, s = math.cos(theta / 2), 1j * math.sin(theta / 2)
    for i in range(n):
        v = psi.view(-1, 2, 1 << i)
        a = v[:, 0] * c
        a += v[:, 1] * s
        v[:, 1].mul_(c)
        v[:, 1].add_(v[:, 0], alpha=s)
        v[:, 0].copy_(a)
        del a
    psi *= complex(math.cos(n * theta / 2), -math.sin(n * theta / 2))


def _strang(psi, n, E, dts, ss):
    """Strang steps of lengths dts frozen at ss; adjacent half phases merged."""
    half = 0.0
    for dt, s in zip(dts, ss):
        _phase(psi, E, half + 0.5 * dt * s)
        _mix(psi, n, dt * (1.0 - s))
        half = 0.5 * dt * s
    _phase(psi, E, half)


def _steps_of(case):
    K = case["steps"]
    dt = case["T"] / K
    if case["call"] == "schedule":
        return [dt] * K, _sweep(case).tolist()
    if case["call"] == "order4":
        w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
        dts, ss = [], []
        for k in range(K):
            t = k * dt
            for w in (w1, 1.0 - 2.0 * w1, w1):
                dts.append(w * dt)
                ss.append((t + 0.5 * w * dt) / case["T"])
                t += w * dt
        return dts, ss
    ks = range(case.get("k0", 0), case.get("k1", K))
    return [dt] * len(ks), [(k + 0.5) / K for k in ks]


def _observables(psi, n, E):
    part = 1 << min(n, 24)
    norm = hp = ground = corr = 0.0
    count = 0
    for i in range(0, 1 << n, part):
        p = torch.view_as_real(psi[i : i + part].to(torch.complex128)).square().sum(-1)
        e = E[i : i + part]
        norm += float(p.sum())
        hp += float((p * e).sum())
        ground += float(p[e == 0].sum())
        count += int((e == 0).sum())
    for b in range(n):
        v = torch.view_as_real(psi).view(-1, 2, 2 << b)
        rows = max(1, part >> b)
        for j in range(0, v.shape[0], rows):
            for k in range(0, 2 << b, part):
                w = v[j : j + rows, :, k : k + part].double()
                corr += float((w[:, 0] * w[:, 1]).sum())
    return {"norm": norm, "expect_hp": hp, "expect_hb": 0.5 * n * norm - corr, "ground_prob": ground, "ground_count": count}


def _levels(n, E, s, levels, iters):
    """The lowest levels reached from the uniform state: Lanczos with full reorthogonalisation in 64 bits."""
    N = 1 << n
    v = torch.full((N,), 2.0 ** (-0.5 * n), dtype=torch.float64, device=E.device)
    V, alpha, beta = [v], [], []
    Ed = E.double()
    for _ in range(iters):
        v = V[-1]
        w = (0.5 * n * (1.0 - s) + s * Ed) * v
        for b in range(n):
            w -= (0.5 * (1.0 - s)) * v.view(-1, 2, 1 << b).flip(1).reshape(-1)
        alpha.append(float(v @ w))
        M = torch.stack(V)
        for _ in range(2):
            w -= (M @ w) @ M
        del M
        b = float(w.norm())
        if b < 1e-10:
            break
        beta.append(b)
        V.append(w / b)
    k = len(alpha)
    T = np.diag(alpha) + np.diag(beta[: k - 1], 1) + np.diag(beta[: k - 1], -1)
    return np.linalg.eigvalsh(T)[:levels]


def exact(case, seed):
    if case["call"] == "serve":
        return None  # hundreds of thousands of steps in all
    n = case["n"]
    clauses = _planted(n, case["m"], np.random.default_rng([seed, n]))
    E = _energies(n, clauses)
    if case["call"] == "spectrum":
        if n > 21:
            return None  # the kept vectors are too many
        levels = _levels(n, E, case["s"], case["levels"], case["iters"])
        return {"levels": levels.tolist(), "iters": None}
    if case["call"] == "observe":
        return _observables(_mid_run_state(n, seed), n, E)
    if case["call"] == "resume":
        psi = _mid_run_state(n, seed).to(torch.complex128)
    else:
        psi = torch.full((1 << n,), 2.0 ** (-0.5 * n), dtype=torch.complex128, device=_device())
    _strang(psi, n, E, *_steps_of(case))
    return {"psi": psi, "observables": _observables(psi, n, E)}
