"""The workloads whose speed is measured, each through the package's public entry points.

A case is one pass of a program that keeps its cost vector, statistics, workspace and state buffers from pass to
pass, as qaoa.optimize does: a training step (objective and gradient), a simulation, a sampling pass, an XY-mixer
simulation, or the build of a cost vector.  Sizes run from states that fit one SM to the 2^30 amplitudes of the
headline workload; problems are those of inputs.py (LABS, weighted MaxCut) and random polynomials with odd orders.
"""
import math

import numpy as np
import torch

from paper_2309_04841_gb300 import inputs
from paper_2309_04841_gb300 import qaoa as Q

STATE = {"c64": Q.C64, "c128": Q.C128}
COST = {"i32": Q.COST_I32, "f32": Q.COST_F32, "u16": Q.COST_U16}


def listed():
    return [
        # the smallest optimizer step: a toy LABS instance, where a call is latency
        dict(name="train_labs10", kind="train", problem="labs", n=10, p=12, cost="i32", state="c64"),
        # the 3-regular MaxCut instance of the tests and the benchmark, in double precision
        dict(name="train_maxcut14_c128", kind="train", problem="maxcut", n=14, p=2, cost="i32", state="c128"),
        # a request of the serving stream: mid-size, deep circuit
        dict(name="train_labs18", kind="train", problem="labs", n=18, p=20, cost="i32", state="c64"),
        # a polynomial with linear and cubic terms (fields), mid-size, an odd number of qubits
        dict(name="train_poly23", kind="train", problem="poly", n=23, p=8, cost="i32", state="c64"),
        # the weighted Erdos-Renyi instance: forward simulation with energy and overlap, real costs
        dict(name="simulate_gnp26", kind="simulate", problem="gnp", n=26, p=6, cost="f32", state="c64"),
        # reference precision on a mid-size LABS instance
        dict(name="train_labs23_c128", kind="train", problem="labs", n=23, p=4, cost="i32", state="c128"),
        # sampling from a trained circuit: state and probabilities, compact costs
        dict(name="sample_labs27_u16", kind="sample", problem="labs", n=27, p=6, cost="u16", state="c64"),
        # the deep gradient workload, weighted MaxCut
        dict(name="train_maxcut28", kind="train", problem="maxcut", n=28, p=20, cost="f32", state="c64"),
        # the headline: LABS n = 30, p = 10, objective and all 20 derivatives
        dict(name="train_labs30", kind="train", problem="labs", n=30, p=10, cost="i32", state="c64"),
        # Hamming-weight-preserving mixers from a Dicke state
        dict(name="xy_ring25", kind="xy", problem="labs", n=25, p=4, cost="i32", state="c64", graph="ring"),
        dict(name="xy_complete19", kind="xy", problem="gnp", n=19, p=2, cost="f32", state="c64", graph="complete"),
        # a new problem instance: its cost vector from the polynomial's terms, and its statistics
        dict(name="costs_poly24", kind="costs", problem="poly4", n=24, p=0, cost="i32", state="c64"),
    ]


def draw(rng):
    kind = rng.choice(["train", "train", "train", "simulate", "sample", "xy", "costs"])
    p = int(round(math.exp(rng.uniform(0.0, math.log(40)))))
    if kind == "costs":
        problem = rng.choice(["poly4", "poly", "maxcut"])
        cost = rng.choice(["i32", "f32"])
        n = rng.randint(8, 26)
        return dict(kind=kind, problem=problem, n=n + n % 2 if problem == "maxcut" else n, p=0, cost=cost, state="c64")
    if kind == "xy":
        graph = rng.choice(["ring", "complete"])
        n = rng.randint(6, 27 if graph == "ring" else 20)
        return dict(kind=kind, problem=rng.choice(["labs", "gnp"]), n=n, p=1 + p % 5, cost=rng.choice(["i32", "f32"]),
                    state="c64", graph=graph)
    state = rng.choice(["c64", "c64", "c128"])
    problem = rng.choice(["labs", "labs", "maxcut", "gnp", "poly"])
    n = rng.randint(4, 29 if state == "c64" else 23)
    if problem == "maxcut":
        n += n % 2
    if problem == "labs":
        cost = rng.choice(["i32", "i32", "u16"])
    else:
        cost = rng.choice(["i32", "f32"]) if problem != "gnp" else "f32"
    # no more work than the headline: fewer layers where the state is large
    if state == "c64":
        p = min(p, 40 if n <= 27 else 20 if n == 28 else 10)
    else:
        p = min(p, 8 if n <= 20 else 3)
    return dict(kind=kind, problem=problem, n=n, p=p, cost=cost, state=state)


# ------------------------------------------------------------------ inputs

def _angles(case, seed):
    """LABS costs are large integers, so the gammas in use are small."""
    ghi = 0.1 if case["problem"] == "labs" else 0.6
    return (inputs.angles(case["p"], 1000 + 7 * seed, 0.0, ghi), inputs.angles(case["p"], 2003 + 7 * seed, 0.0, math.pi))


def _edges(case, seed):
    """(edges, weights) of the case's graph; integer weights for integer costs."""
    n = case["n"]
    if case["problem"] == "maxcut":
        e, w = inputs.maxcut_3reg(n, graph_seed=1 + seed, weighted=True, weight_seed=4 + seed)
    else:
        e, w = inputs.maxcut_gnp(n, 0.5, graph_seed=3 + seed, weight_seed=4 + seed)
    return e, (np.floor(w * 8) + 1 if case["cost"] == "i32" else w)


def _terms(case, seed):
    """Random polynomial of orders 0..4 ("poly": about 4 n terms, linear ones among them; "poly4": the dense
    instances, about n^2 terms).  Integer weights, or multiples of 2^-20 for real costs."""
    n = case["n"]
    count = 4 * n if case["problem"] == "poly" else min(n * n, 1000)
    return inputs.random_terms(n, count, 11 + seed, max_order=4, integer=case["cost"] == "i32")


def _costs(case, seed):
    n, kind = case["n"], case["cost"]
    if case["problem"] == "labs":
        return Q.labs_costs_u16(n) if kind == "u16" else Q.labs_costs(n) if kind == "i32" else Q.labs_costs(n).to(torch.float32)
    if case["problem"] in ("maxcut", "gnp"):
        e, w = _edges(case, seed)
        return Q.maxcut_costs(n, e, w, COST[kind])
    return Q.precompute_costs(n, Q.terms_array(_terms(case, seed)), COST[kind])


def prepare(case, seed):
    n, s = case["n"], dict(case)
    s["work"] = Q.workspace(n)
    if case["kind"] == "costs":
        if case["problem"] == "maxcut":
            s["edges"], s["weights"] = _edges(case, seed)
        else:
            s["terms"] = Q.terms_array(_terms(case, seed))
        s["costs"] = torch.empty(1 << n, dtype=Q.cost_dtype(COST[case["cost"]]), device="cuda")
        return s
    s["gammas"], s["betas"] = _angles(case, seed)
    s["costs"] = _costs(case, seed)
    s["stats"] = Q.cost_stats_compute(s["costs"], work=s["work"])
    s["state"] = torch.empty(1 << n, dtype=Q.state_dtype(STATE[case["state"]]), device="cuda")
    if case["kind"] == "train":
        s["lam"] = torch.empty_like(s["state"])
        s["out"] = torch.empty(2 + 2 * case["p"], dtype=torch.float64, device="cuda")
    elif case["kind"] == "sample":
        s["probs"] = torch.empty(1 << n, dtype=torch.float32 if case["state"] == "c64" else torch.float64, device="cuda")
    else:
        s["out"] = torch.empty(2, dtype=torch.float64, device="cuda")
    return s


# -------------------------------------------------------------------- runs

def _real(s, v):
    """Results in the precision of the state: single-precision states train single-precision parameters."""
    return v.to(torch.float32) if s["state"].dtype == torch.complex64 else v


def run(s):
    kind = s["kind"]
    if kind == "costs":
        if "edges" in s:
            Q.maxcut_costs(s["n"], s["edges"], s["weights"], COST[s["cost"]], out=s["costs"])
        else:
            Q.precompute_costs(s["n"], s["terms"], COST[s["cost"]], out=s["costs"])
        st = Q.cost_stats_compute(s["costs"], work=s["work"])
        return {"costs": s["costs"], "f_min": st.f_min, "f_max": st.f_max, "n_min": int(st.n_min), "step": int(st.step_log2)}
    if kind == "train":
        v = _real(s, Q.grad(s["costs"], s["stats"], s["gammas"], s["betas"], state=s["state"], lam=s["lam"],
                            state_type=Q.state_type_of(s["state"]), work=s["work"], out=s["out"]))
        return {"value": v[:2], "grad": v[2:]}
    if kind == "simulate":
        state, out = Q.simulate(s["costs"], s["stats"], s["gammas"], s["betas"], state=s["state"],
                                state_type=Q.state_type_of(s["state"]), work=s["work"], out=s["out"])
        return {"state": state, "value": _real(s, out)}
    if kind == "sample":
        state, _ = Q.simulate(s["costs"], s["stats"], s["gammas"], s["betas"], state=s["state"],
                              state_type=Q.state_type_of(s["state"]), work=s["work"], reduce=False)
        return {"state": state, "probs": Q.probabilities(state, out=s["probs"])}
    state = Q.dicke_state(s["n"], s["n"] // 2, out=s["state"])
    state, out = Q.simulate_xy(s["costs"], s["stats"], s["gammas"], s["betas"], state,
                               graph=Q.XY_RING if s["graph"] == "ring" else Q.XY_COMPLETE, work=s["work"], out=s["out"])
    return {"state": state, "value": _real(s, out)}


def work(case):
    """Inputs read once, outputs written once; the rotations and phases of every layer."""
    n, p, N = case["n"], case["p"], float(1 << case["n"])
    cb = {"i32": 4, "f32": 4, "u16": 2}[case["cost"]]
    sb = 8 if case["state"] == "c64" else 16
    if case["kind"] == "costs":
        terms = 1.5 * n if case["problem"] == "maxcut" else 4 * n if case["problem"] == "poly" else min(n * n, 1000)
        return {"bytes": cb * N, "flops": terms + n * N}  # a fast Walsh-Hadamard transform: n additions an element
    layer = 4.0 * n * N + 8.0 * N  # n / 2 pairs an amplitude at 8 operations, one complex product
    if case["kind"] == "train":
        return {"bytes": cb * N + 8.0 * (2 + 2 * p), "flops": 4.0 * p * layer}
    if case["kind"] == "sample":
        return {"bytes": (cb + sb + sb / 2) * N, "flops": p * layer}
    if case["kind"] == "xy":
        gates = n if case["graph"] == "ring" else n * (n - 1) / 2
        return {"bytes": (cb + sb) * N, "flops": p * (4.0 * gates * N + 8.0 * N)}
    return {"bytes": (cb + sb) * N, "flops": p * layer}


# ------------------------------------------------------------------- exact
# The same results in 64 bits: costs from their definitions, gates one at a time.

def _popcount(v):
    """Bits set in each element of an int64 tensor below 2^32."""
    v = v - ((v >> 1) & 0x55555555)
    v = (v & 0x33333333) + ((v >> 2) & 0x33333333)
    v = (v + (v >> 4)) & 0x0F0F0F0F
    return (((v * 0x01010101) & 0xFFFFFFFF) >> 24)


def _exact_costs(case, seed):
    """float64 cost vector, in blocks of 2^24 elements."""
    n = case["n"]
    f = torch.empty(1 << n, dtype=torch.float64, device="cuda")
    step = 1 << min(n, 24)
    if case["problem"] in ("maxcut", "gnp"):
        e, w = _edges(case, seed)
        e, w = e.tolist(), w.tolist()
    elif case["problem"] != "labs":
        terms = [(float(w), sum(1 << i for i in idx)) for w, idx in _terms(case, seed)]
    for x0 in range(0, 1 << n, step):
        x = torch.arange(x0, x0 + step, dtype=torch.int64, device="cuda")
        g = torch.zeros(step, dtype=torch.float64, device="cuda")
        if case["problem"] == "labs":
            for k in range(1, n):
                c = (n - k) - 2 * _popcount((x ^ (x >> k)) & ((1 << (n - k)) - 1))
                g += (c * c).to(torch.float64)
        elif case["problem"] in ("maxcut", "gnp"):
            for (i, j), wij in zip(e, w):
                g -= wij * (((x >> i) ^ (x >> j)) & 1).to(torch.float64)
        else:
            for w, mask in terms:
                g += w * (1 - 2 * (_popcount(x & mask) & 1)).to(torch.float64)
        f[x0:x0 + step] = g
    return f


def _phase(psi, f, gamma):
    step = 1 << 26
    for x in range(0, psi.numel(), step):
        a = f[x:x + step] * gamma
        psi[x:x + step] *= torch.complex(torch.cos(a), -torch.sin(a))


def _mix(psi, tmp, n, beta):
    """exp(-i beta sum X) psi, with the scale of the reduced gates put back at the end; returns (result, spare)."""
    c, s = math.cos(beta), math.sin(beta)
    for q in range(n):
        a, b = psi.view(-1, 2, 1 << q).unbind(1)
        u, v = tmp.view(-1, 2, 1 << q).unbind(1)
        if abs(c) >= abs(s):
            torch.add(a, b, alpha=-1j * s / c, out=u)
            torch.add(b, a, alpha=-1j * s / c, out=v)
        else:
            torch.add(b, a, alpha=1j * c / s, out=u)
            torch.add(a, b, alpha=1j * c / s, out=v)
        psi, tmp = tmp, psi
    psi *= (c if abs(c) >= abs(s) else -1j * s) ** n
    return psi, tmp


def _value(psi, f, f_min):
    e = o = 0.0
    step = 1 << 26
    for x in range(0, psi.numel(), step):
        pr = psi[x:x + step].abs().square()
        e += float((pr * f[x:x + step]).sum())
        o += float(pr[f[x:x + step] == f_min].sum())
    return torch.tensor([e, o], dtype=torch.float64)


def exact(case, seed):
    n, p = case["n"], case["p"]
    f = _exact_costs(case, seed)
    if case["kind"] == "costs":
        return {"costs": f if case["cost"] == "f32" else None, "f_min": float(f.min()), "f_max": float(f.max()),
                "n_min": None, "step": None}
    gammas, betas = _angles(case, seed)
    f_min = float(f.min())
    N = 1 << n
    if case["kind"] == "xy":
        psi = torch.zeros(N, dtype=torch.complex128, device="cuda")
        x = torch.arange(N, dtype=torch.int64, device="cuda")
        psi[_popcount(x) == n // 2] = 1.0 / math.sqrt(math.comb(n, n // 2))
        if case["graph"] == "ring":
            edges = [(q, q + 1) for q in range(n - 1)] + ([(0, n - 1)] if n >= 3 else [])
        else:
            edges = [(i, j) for i in range(n) for j in range(i + 1, n)]
        for g, b in zip(gammas, betas):
            _phase(psi, f, g)
            for i, j in edges:
                v = psi.view(-1, 2, 1 << (j - i - 1), 2, 1 << i)
                u, w = v[:, 0, :, 1], v[:, 1, :, 0]
                t = math.cos(b) * u - 1j * math.sin(b) * w
                w.copy_(math.cos(b) * w - 1j * math.sin(b) * u)
                u.copy_(t)
        return {"state": psi, "value": _value(psi, f, f_min)}
    psi = torch.full((N,), 1.0 / math.sqrt(N), dtype=torch.complex128, device="cuda")
    tmp = torch.empty_like(psi)
    for g, b in zip(gammas, betas):
        _phase(psi, f, g)
        psi, tmp = _mix(psi, tmp, n, b)
    if case["kind"] == "sample":
        del tmp
        return {"state": psi, "probs": psi.abs().square()}
    value = _value(psi, f, f_min)
    if case["kind"] == "simulate":
        return {"state": psi, "value": value}
    if n * float(N) * p > 30 * 2.0 ** 28 * 20:  # over the time that a gate-by-gate gradient may take
        return {"value": value, "grad": None}
    lam = psi * f
    dg, db = [0.0] * p, [0.0] * p
    for k in range(p - 1, -1, -1):
        tmp.zero_()
        for q in range(n):
            a, b = psi.view(-1, 2, 1 << q).unbind(1)
            u, v = tmp.view(-1, 2, 1 << q).unbind(1)
            u += b
            v += a
        db[k] = 2 * float(torch.vdot(lam, tmp).imag)
        psi, tmp = _mix(psi, tmp, n, -betas[k])
        lam, tmp = _mix(lam, tmp, n, -betas[k])
        torch.mul(psi, f, out=tmp)
        dg[k] = 2 * float(torch.vdot(lam, tmp).imag)
        _phase(psi, f, -gammas[k])
        _phase(lam, f, -gammas[k])
    return {"value": value, "grad": torch.tensor(dg + db, dtype=torch.float64)}
