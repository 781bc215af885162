"""Timed workloads of the library: what its users have it do, through its public
entry points, from the smallest call to the largest.

Each case is one operation:

* ``whole``   clauses in, amplitudes and success probability out, one instance
              (``api.psucc_host``: cost table, evolution, fused reduction);
* ``tables``  a batch of instances of one n: their cost tables, then their
              evolutions with shared angles (``api.cost_table_batch``,
              ``api.evolve_batch``), as the instance studies run them;
* ``half``    the batched evolution on the halved state, the tables in hand
              (``api.evolve_batch`` with ``Z2_HALF``), as the scaling sweep runs it;
* ``running`` bitstrings drawn from a batch of output states until one satisfies
              (``api.running_time_batch``);
* ``grad``    batched gradients with shared angles, the tables in hand, one step
              of angle training (``api.grad_batch``);
* ``serve``   a burst of requests of uneven n and p through the serving loop
              (``serve.Server``), submitted together and waited for.

Arithmetic: ``c64``, ``c128`` (FP64) and ``df64`` (complex128 held in
double-float pairs).  Figures reduced from a complex64 state (success
probabilities, norms, gradients) are handed on as float32, the precision of the
amplitudes they come from; those of complex128 states as float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2401_02852_gb300 import api, serve
from paper_2401_02852_gb300.instances import Instance, Request

FLAGS = {"c64": 0, "c128": 0, "df64": api._lib.DF64}
DTYPE = {"c64": "c64", "c128": "c128", "df64": "c128"}


def listed():
    return [
        # the smallest use: one n = 12 NAE-3-SAT instance (m = 24, p = 5), FP64;
        # launches, copies and one instance's latency count
        {"name": "whole_n12_c128", "op": "whole", "n": 12, "k": 3, "r": 2.0, "p": 5, "arith": "c128"},
        # an ordinary request, its state resident in L2, odd n and p
        {"name": "whole_n21_c64", "op": "whole", "n": 21, "k": 5, "r": 8.0, "p": 7, "arith": "c64"},
        # the large single state of the precision study (8.6 GB)
        {"name": "whole_n30_c64", "op": "whole", "n": 30, "k": 5, "r": 8.0, "p": 10, "arith": "c64"},
        # the study's FP64 arm at a size a user iterates on
        {"name": "whole_n26_c128", "op": "whole", "n": 26, "k": 5, "r": 8.0, "p": 10, "arith": "c128"},
        # its double-float arm
        {"name": "whole_n27_df64", "op": "whole", "n": 27, "k": 5, "r": 8.0, "p": 10, "arith": "df64"},
        # 100 small FP64 instances, tables and evolutions
        {"name": "tables_n12_x100_c128", "op": "tables", "n": 12, "k": 3, "r": 2.0, "p": 5, "batch": 100,
         "arith": "c128"},
        # the paper's evaluation at the threshold density of k = 9 (about 3000 clauses)
        {"name": "tables_n17_k9_x256_c64", "op": "tables", "n": 17, "k": 9, "r": 176.85, "p": 8, "batch": 256,
         "arith": "c64"},
        # the scaling sweep's batched evolutions on the halved state
        {"name": "half_n24_x24_c64", "op": "half", "n": 24, "k": 5, "r": 8.0, "p": 10, "batch": 24, "arith": "c64"},
        # running times of a batch of evaluation states
        {"name": "running_n19_x256_c64", "op": "running", "n": 19, "k": 9, "r": 176.85, "p": 4, "batch": 256,
         "draws": 4096, "arith": "c64"},
        # shared-angle training on n = 22 instances, deep circuits
        {"name": "grad_n22_x32_c64", "op": "grad", "n": 22, "k": 5, "r": 8.0, "p": 20, "batch": 32, "arith": "c64"},
        # the paper's training step: 100 instances of n = 12 in FP64
        {"name": "grad_n12_x100_c128", "op": "grad", "n": 12, "k": 5, "r": 10.494, "p": 16, "batch": 100,
         "arith": "c128"},
        # a burst of the serving stream: n in 14..26, p in 1..20
        {"name": "serve_x48_c64", "op": "serve", "n": 14, "n_max": 26, "k": 5, "r": 8.0, "p": 20, "batch": 48,
         "arith": "c64"},
    ]


# Amplitude-layers a drawn case may have (times its instances): no more than the
# largest listed case of the same arithmetic.
MOST = {"c64": 10 << 30, "c128": 10 << 26, "df64": 10 << 27}


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["whole", "whole", "tables", "tables", "half", "running", "grad", "grad", "serve"])
    p = _log_int(rng, 1, 20)
    if op == "whole":
        arith = rng.choice(["c64", "c64", "c128", "df64"])
        n = rng.randint(10, {"c64": 30, "c128": 26, "df64": 27}[arith])
        while (p << n) > MOST[arith]:
            p -= 1
        k, r = (3, 2.0) if n < 14 else (5, 8.0)
        return {"op": op, "n": n, "k": k, "r": r, "p": p, "arith": arith}
    if op == "tables":
        n = rng.randint(10, 19)
        k, r = rng.choice([(3, 2.0), (5, 10.494), (7, 43.765), (9, 176.85)])
        arith = rng.choice(["c64", "c64", "c128", "df64"]) if n <= 14 else "c64"
        return {"op": op, "n": n, "k": k, "r": r, "p": p, "batch": _log_int(rng, 16, min(512, 1 << (26 - n))),
                "arith": arith}
    if op == "half":
        n = rng.randint(16, 27)
        return {"op": op, "n": n, "k": 5, "r": 8.0, "p": p, "batch": _log_int(rng, 1, min(200, 1 << (29 - n))),
                "arith": "c64"}
    if op == "running":
        n = rng.randint(12, 20)
        return {"op": op, "n": n, "k": 7, "r": 43.765, "p": rng.randint(1, 4),
                "batch": _log_int(rng, 8, min(512, 1 << (27 - n))), "draws": _log_int(rng, 1000, 16384),
                "arith": rng.choice(["c64", "c64", "c64", "c128"])}
    if op == "grad":
        if rng.random() < 0.5:
            return {"op": op, "n": rng.randint(10, 12), "k": rng.choice([3, 5]), "r": 8.0, "p": p,
                    "batch": _log_int(rng, 32, 128), "arith": "c128"}
        n = rng.randint(13, 24)
        return {"op": op, "n": n, "k": 5, "r": 8.0, "p": p, "batch": _log_int(rng, 1, min(64, 1 << (27 - n))),
                "arith": "c64"}
    return {"op": "serve", "n": rng.randint(10, 16), "n_max": rng.randint(18, 26), "k": 5, "r": 8.0, "p": p,
            "batch": _log_int(rng, 12, 48), "arith": "c64"}


# ---- inputs -------------------------------------------------------------------
def _instance(n, k, m, rng):
    """m clauses: k distinct variables each (the k smallest of n uniform keys),
    fair negations."""
    var = np.argsort(rng.random((m, n)), axis=1)[:, :k].astype(np.int32)
    return Instance(n=n, k=k, var=np.ascontiguousarray(var), neg=rng.integers(0, 2, size=(m, k), dtype=np.uint8))


def _instances(case, seed):
    """The case's instances; clause counts fixed at round(r n), or Poisson
    around r n at the long lists of the evaluation."""
    n, k, r = case["n"], case["k"], case["r"]
    out = []
    for b in range(case.get("batch", 1)):
        rng = np.random.default_rng([int(seed), n, k, b])
        m = int(rng.poisson(r * n)) if r > 10 else int(round(r * n))
        out.append(_instance(n, k, m, rng))
    return out


def _ramp(p):
    l = np.arange(1, p + 1, dtype=np.float64)
    return 0.8 * (l - 0.5) / p, 0.8 * (1.0 - (l - 0.5) / p)


def _angles(case, seed):
    """Linear-ramp angles; in training they have moved off the ramp."""
    g, b = _ramp(case["p"])
    if case["op"] == "grad":
        rng = np.random.default_rng([int(seed), 77])
        g, b = g + 0.02 * rng.standard_normal(g.size), b + 0.02 * rng.standard_normal(b.size)
    return g, b


def _requests(case, seed):
    """Requests of uneven size, spread evenly over n .. n_max and 1 .. p in a
    seeded order, so that a burst of any seed is about the same work."""
    rng = np.random.default_rng([int(seed), 5])
    count, lo, hi = case["batch"], case["n"], case["n_max"]
    ns = [lo + (i * (hi - lo + 1)) // count for i in range(count)]
    out = []
    for i in rng.permutation(count):
        n = ns[i]
        p = 1 + int((i * 0.6180339887498949) % 1.0 * case["p"])
        g, b = _ramp(p)
        out.append(Request(_instance(n, case["k"], int(round(case["r"] * n)), rng), p, g, b, 0.0))
    return out


class _Serving:
    """A server and a burst for it; the server closes with its owner."""

    def __init__(self, case, seed):
        self.requests = _requests(case, seed)
        self.server = serve.Server(case["arith"], hbm_budget_bytes=8 << 30)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    if case["op"] == "serve":
        return {"case": case, "serving": _Serving(case, seed)}
    n, arith = case["n"], case["arith"]
    tdt = torch.complex64 if arith == "c64" else torch.complex128
    insts = _instances(case, seed)
    gamma, beta = _angles(case, seed)
    st = {"case": case, "gamma": gamma, "beta": beta, "insts": insts, "m": max(i.m for i in insts)}
    B = len(insts)
    if case["op"] == "whole":
        st["work"] = {"cost": torch.empty(1 << n, dtype=torch.uint8, device="cuda"),
                      "state": torch.empty(1 << n, dtype=tdt, device="cuda")}
    elif case["op"] == "tables":
        st["costs"] = torch.empty((B, 1 << n), dtype=torch.uint8, device="cuda")
        st["states"] = torch.empty((B, 1 << n), dtype=tdt, device="cuda")
    elif case["op"] == "half":
        st["costs"] = torch.empty((B, 1 << (n - 1)), dtype=torch.uint8, device="cuda")
        for b, inst in enumerate(insts):
            api.cost_table_half(inst, out=st["costs"][b], stats=False)
        st["states"] = torch.empty((B, 1 << (n - 1)), dtype=tdt, device="cuda")
    elif case["op"] == "running":
        st["costs"] = api.cost_table_batch(insts)[0]
        st["states"] = _evolve_plain(st["costs"], gamma, beta, tdt)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        st["u"] = torch.rand((B, case["draws"]), dtype=torch.float64, device="cuda", generator=gen)
    else:
        st["costs"] = api.cost_table_batch(insts)[0]
        st["work"] = tuple(torch.empty((B, 1 << n), dtype=tdt, device="cuda") for _ in range(2))
    return st


def _figures(arith, *values):
    """Reduced figures in the real type of the state they come from."""
    dt = np.float32 if arith == "c64" else np.float64
    return [np.asarray(v, dtype=dt) for v in values]


def run(st):
    case = st["case"]
    op, arith = case["op"], case["arith"]
    if op == "serve":
        s = st["serving"]
        tickets = [s.server.submit(r.instance, r.gamma, r.beta) for r in s.requests]
        res = [s.server.wait(t) for t in tickets]
        ps, nm = _figures(arith, [r.p_succ for r in res], [r.norm for r in res])
        return {"p_succ": ps, "norm": nm, "n_sol": np.array([r.n_sol for r in res]),
                "max_cost": np.array([r.max_cost for r in res]), "status": np.array([r.status for r in res])}
    n, g, b = case["n"], st["gamma"], st["beta"]
    if op == "whole":
        ps, nm = api.psucc_host(st["insts"][0], g, b, DTYPE[arith], flags=FLAGS[arith], work=st["work"])
        ps, nm = _figures(arith, ps, nm)
        return {"p_succ": ps, "norm": nm, "state": st["work"]["state"], "cost": st["work"]["cost"]}
    if op == "tables":
        costs, sols, mx = api.cost_table_batch(st["insts"], out=st["costs"])
        states, ps, nm = api.evolve_batch(n, costs, st["m"], g, b, DTYPE[arith], flags=FLAGS[arith],
                                          out=st["states"])
        ps, nm = _figures(arith, ps, nm)
        return {"p_succ": ps, "norm": nm, "n_sol": sols, "max_cost": mx, "state": states, "cost": costs}
    if op == "half":
        states, ps, nm = api.evolve_batch(n, st["costs"], st["m"], g, b, DTYPE[arith], flags=api.Z2_HALF,
                                          out=st["states"])
        ps, nm = _figures(arith, ps, nm)
        return {"p_succ": ps, "norm": nm, "state": states}
    if op == "running":
        return {"running_time": api.running_time_batch(n, st["costs"], st["states"], st["u"])}
    ps, dg, db = api.grad_batch(n, st["costs"], st["m"], g, b, DTYPE[arith], work=st["work"])
    ps, dg, db = _figures(arith, ps, dg, db)
    return {"p_succ": ps, "dgamma": dg, "dbeta": db}


# ---- what a pass cannot do without -----------------------------------------------
def work(case):
    """Inputs read once, outputs written once; floating operations of the layers
    (two multiply-adds per amplitude and qubit, a complex product per phase)."""
    op, n, p = case["op"], case["n"], case["p"]
    es = 8 if case["arith"] == "c64" else 16
    if op == "serve":
        # the requests' (n, p) do not depend on the seed; results are a few bytes each
        amp = sum((1 << r.instance.n) * r.p * (4 * r.instance.n + 6) for r in _requests(case, 0))
        return {"bytes": float(sum(r.instance.var.nbytes + r.instance.neg.nbytes + 48 for r in _requests(case, 0))),
                "flops": float(amp)}
    B, N = case.get("batch", 1), 1 << n
    m = int(round(case["r"] * n))
    clauses = B * m * case["k"] * 5
    layers = float(B) * N * p * (4 * n + 6)
    if op in ("whole", "tables"):
        return {"bytes": float(clauses + B * N * (1 + es)), "flops": layers}
    if op == "half":
        return {"bytes": float(B * (N // 2) * (1 + es)), "flops": layers / 2}
    if op == "running":
        return {"bytes": float(B * (N * es + case["draws"] * 8)), "flops": float(B * N * 3)}
    return {"bytes": float(B * N), "flops": 4 * layers}


# ---- the same results in plain torch, 64 bits --------------------------------------
def _cost_plain(inst):
    """C(x) of one instance: clauses whose literals are all equal."""
    n = inst.n
    mask = np.zeros(inst.m, dtype=np.int64)
    neg = np.zeros(inst.m, dtype=np.int64)
    for j in range(inst.k):
        mask |= np.int64(1) << inst.var[:, j].astype(np.int64)
        neg |= inst.neg[:, j].astype(np.int64) << inst.var[:, j].astype(np.int64)
    mask_d = torch.from_numpy(mask).to(torch.int32).cuda()
    neg_d = torch.from_numpy(neg).to(torch.int32).cuda()
    out = torch.empty(1 << n, dtype=torch.int32, device="cuda")
    step = min(1 << n, 1 << 22)
    rows = max(1, (1 << 27) // step)
    for x0 in range(0, 1 << n, step):
        x = torch.arange(x0, x0 + step, dtype=torch.int32, device="cuda")
        acc = torch.zeros(step, dtype=torch.int32, device="cuda")
        for i in range(0, inst.m, rows):
            mk, ng = mask_d[i:i + rows, None], neg_d[i:i + rows, None]
            t = (x[None, :] ^ ng) & mk
            acc += ((t == 0) | (t == mk)).sum(0, dtype=torch.int32)
        out[x0:x0 + step] = acc
    return out


def _costs_plain(insts):
    return torch.stack([_cost_plain(i) for i in insts])


def _mix_plain(psi, beta):
    """prod_j [cos(beta) I + i sin(beta) X_j] on [B, 2^n] (returned; psi is used up)."""
    B, N = psi.shape
    c, s = math.cos(beta), math.sin(beta)
    buf = torch.empty_like(psi)
    for j in range(N.bit_length() - 1):
        v, w = psi.view(B, -1, 2, 1 << j), buf.view(B, -1, 2, 1 << j)
        torch.mul(v, c, out=w)
        w[:, :, 0].add_(v[:, :, 1], alpha=1j * s)
        w[:, :, 1].add_(v[:, :, 0], alpha=1j * s)
        psi, buf = buf, psi
    return psi


def _phase_plain(psi, costs, gamma):
    """psi exp(-i gamma C), by a table over the values of C."""
    c = torch.arange(int(costs.max()) + 1, dtype=torch.float64, device="cuda")
    tab = torch.complex(torch.cos(gamma * c), -torch.sin(gamma * c)).to(psi.dtype)
    step = 1 << 28
    flat, fc = psi.view(-1), costs.reshape(-1)
    for x0 in range(0, flat.numel(), step):
        flat[x0:x0 + step] *= tab[fc[x0:x0 + step].long()]
    return psi


def _evolve_plain(costs, gamma, beta, tdt=torch.complex128):
    B, N = costs.shape
    psi = torch.full((B, N), 1.0 / math.sqrt(N), dtype=tdt, device="cuda")
    for g, b in zip(gamma, beta):
        psi = _mix_plain(_phase_plain(psi, costs, float(g)), float(b))
    return psi


def _sums_plain(costs, psi):
    w = psi.real.square() + psi.imag.square()
    return (w * (costs == 0)).sum(1).cpu().numpy(), w.sum(1).cpu().numpy()


def _grad_plain(costs, gamma, beta):
    """p_succ and its derivatives, layers undone backward on (psi, lam)."""
    B, N = costs.shape
    p = len(gamma)
    psi = _evolve_plain(costs, gamma, beta)
    ps = _sums_plain(costs, psi)[0]
    lam = psi * (costs == 0)
    dg, db = np.zeros((B, p)), np.zeros((B, p))
    fc = costs.double()
    for l in reversed(range(p)):
        acc = torch.zeros(B, dtype=torch.float64, device="cuda")
        for j in range(N.bit_length() - 1):
            v, u = psi.view(B, -1, 2, 1 << j), lam.view(B, -1, 2, 1 << j)
            for h in (0, 1):
                a, o = u[:, :, h], v[:, :, 1 - h]
                acc += (a.real * o.imag - a.imag * o.real).sum((1, 2))
        db[:, l] = -2.0 * acc.cpu().numpy()
        psi, lam = _mix_plain(psi, -float(beta[l])), _mix_plain(lam, -float(beta[l]))
        dg[:, l] = 2.0 * (fc * (lam.real * psi.imag - lam.imag * psi.real)).sum(1).cpu().numpy()
        psi, lam = _phase_plain(psi, costs, -float(gamma[l])), _phase_plain(lam, costs, -float(gamma[l]))
    return ps, dg, db


def exact(case, seed):
    op = case["op"]
    if op == "running":
        return None  # whole numbers
    if op == "serve":
        ps, nm = [], []
        for r in _requests(case, seed):
            costs = _costs_plain([r.instance])
            a, b = _sums_plain(costs, _evolve_plain(costs, r.gamma, r.beta))
            ps.append(a[0])
            nm.append(b[0])
        return {"p_succ": np.array(ps), "norm": np.array(nm), "n_sol": None, "max_cost": None, "status": None}
    insts = _instances(case, seed)
    gamma, beta = _angles(case, seed)
    if op == "grad":
        # the plain reverse sweep takes about 40 passes over a complex128 state per layer and qubit
        if len(insts) * (1 << case["n"]) * case["n"] * case["p"] > (22 * 20) << 27:
            return None
        ps, dg, db = _grad_plain(_costs_plain(insts), gamma, beta)
        return {"p_succ": ps, "dgamma": dg, "dbeta": db}
    costs = _costs_plain(insts)
    psi = _evolve_plain(costs, gamma, beta)
    if op == "half":
        ps, nm = _sums_plain(costs, psi)
        return {"p_succ": ps, "norm": nm, "state": psi[:, :psi.shape[1] // 2].contiguous()}
    if op == "tables":
        ps, nm = _sums_plain(costs, psi)
        return {"p_succ": ps, "norm": nm, "n_sol": None, "max_cost": None, "state": psi, "cost": None}
    ps, nm = _sums_plain(costs, psi)
    return {"p_succ": ps[0], "norm": nm[0], "state": psi[0], "cost": None}
