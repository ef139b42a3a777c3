"""Performance cases: the work a user of this library has it do, through its public calls.

Every case is a dict of plain values.  `kind` says which call it stands for:

  evolve    hs_evolve / hs_evolve_ex on a factor set the program keeps
  anneal    hs_evolve_td of a MaxCut annealing schedule on a kept factor set
  batch     hs_batch_launch of a kept batch of many uneven jobs
  job       one whole request: factor build, evolution, overlap with the start
  apply     hs_apply_factor: one factor application (the paper's Alg. 1)
  dia       hs_dia_evolve: steps of a kept single-factor Taylor propagator (Alg. 3's loop)
  taylor    the whole of Alg. 3: H, step search, propagator, conversion, evolution
  expect    hs_expectation of H on several states

The Hamiltonian families, sizes and budgets are those of the library's workload
module and tests.  The structure of a case (graph, chain, step counts) is fixed by
its fields; couplings and states come from the seed.
"""
import math

import numpy as np
import torch

from paper_2606_16959_gb300 import hs, workloads

BUDGET = {"tfim": 4, "heisenberg": 8, "maxcut": 4, "tsp": 1}


def listed():
    return [
        # The smallest call: the 10-qubit TFIM quick start, ten FP64 steps.  Launches and latency.
        {"name": "tfim10_c128", "kind": "evolve", "family": "tfim", "n": 10, "rhs": 1, "steps": 10, "budget": 4,
         "order": 1, "dtype": "c128", "method": "auto"},
        # The largest spin-chain row of the configurations: one L2-resident state, 100 steps,
        # called as the README does (hs_evolve, no options).
        {"name": "heis16_c64", "kind": "evolve", "family": "heisenberg", "n": 16, "rhs": 1, "steps": 100,
         "budget": 8, "order": 1, "dtype": "c64", "method": "auto"},
        # A higher-order formula in FP64 on an odd chain length with an odd number of states.
        {"name": "heis15_strang_c128", "kind": "evolve", "family": "heisenberg", "n": 15, "rhs": 3, "steps": 20,
         "budget": 8, "order": 2, "dtype": "c128", "method": "auto"},
        # A Heisenberg chain beyond the caches with the register sweep, as served requests run it.
        {"name": "heis22_reg", "kind": "evolve", "family": "heisenberg", "n": 22, "rhs": 2, "steps": 20,
         "budget": 8, "order": 1, "dtype": "c64", "method": "reg"},
        # The headline workload: weighted MaxCut, 24 qubits, 16 states, 50 steps, register sweep.
        {"name": "maxcut24_reg", "kind": "evolve", "family": "maxcut", "n": 24, "rhs": 16, "steps": 50,
         "budget": 4, "order": 1, "dtype": "c64", "method": "reg"},
        # The annealing schedule H(t) = H0 + f(t) H1 at the size of the time-dependent tests.
        {"name": "anneal22_reg", "kind": "anneal", "n": 22, "rhs": 8, "steps": 50, "budget": 4, "dtype": "c64"},
        # An uneven batch of chains, planned once and launched again and again.
        {"name": "batch32", "kind": "batch", "jobs": 32, "n_lo": 12, "n_hi": 20, "steps_lo": 10, "steps_hi": 60,
         "mix": 1004, "dtype": "c64"},
        # One whole request with default options: build the factors, evolve, take the overlap.
        {"name": "job_maxcut20", "kind": "job", "family": "maxcut", "n": 20, "rhs": 4, "steps": 10, "budget": 4,
         "dtype": "c64"},
        # Alg. 1 alone: one stored factor on three states.
        {"name": "apply_heis21", "kind": "apply", "family": "heisenberg", "n": 21, "rhs": 3, "budget": 8, "g": 0,
         "dtype": "c64"},
        # The evolution loop of Alg. 3 with the largest TFIM row's propagator (455 diagonals).
        {"name": "dia_tfim16", "kind": "dia", "n": 16, "rhs": 1, "h": 0.1, "dt": 1.0 / 2088, "steps": 64,
         "dtype": "c64"},
        # The whole of Alg. 3 on a smaller chain: H, budgeted step search, propagator, evolution.
        {"name": "taylor_tfim12", "kind": "taylor", "n": 12, "rhs": 1, "h": 0.1, "budget": 512, "t": 0.25,
         "dtype": "c128"},
        # Energies of several states, as an optimisation loop reads them.
        {"name": "expect_heis20", "kind": "expect", "family": "heisenberg", "n": 20, "rhs": 4, "dtype": "c128"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _even(n):
    return n - (n & 1)


# Amplitudes times terms times steps of the largest listed case: no drawn evolution costs more.
_MOST = 60 * 16 * 50 * (1 << 24)


def draw(rng):
    kind = rng.choice(["evolve", "evolve", "evolve", "anneal", "batch", "job", "apply", "dia", "taylor", "expect"])
    rhs = _log_int(rng, 1, 16)
    if kind == "evolve":
        c = {"kind": kind, "family": rng.choice(["tfim", "heisenberg", "maxcut", "tsp"]), "n": rng.randint(6, 23),
             "rhs": rhs, "steps": _log_int(rng, 5, 100), "budget": 4, "order": rng.choice([1, 1, 2, 4]),
             "dtype": rng.choice(["c64", "c64", "c128"]), "method": rng.choice(["auto", "reg"])}
        if c["family"] == "maxcut":
            c["n"] = _even(c["n"])
        if c["family"] == "tsp":
            c["n"] = 16
        c["budget"] = rng.randint(4, 16) if c["family"] == "heisenberg" else BUDGET[c["family"]]
        c["steps"] = max(2, c["steps"] // {1: 1, 2: 2, 4: 10}[c["order"]])

        def cost():
            f = (20 if c["dtype"] == "c128" else 1) * (6 if c["method"] == "auto" else 3) * {1: 1, 2: 2, 4: 10}[c["order"]]
            return f * 3 * c["n"] * c["rhs"] * c["steps"] * (1 << c["n"])
        while cost() > _MOST and c["rhs"] > 1:
            c["rhs"] = (c["rhs"] + 1) // 2
        while cost() > _MOST and c["steps"] > 2:
            c["steps"] = (c["steps"] + 1) // 2
        while cost() > _MOST and c["family"] != "tsp":
            c["n"] -= 2
        return c
    if kind == "anneal":
        return {"kind": kind, "n": 2 * rng.randint(6, 11), "rhs": min(rhs, 8), "steps": rng.randint(10, 50),
                "budget": 4, "dtype": "c64"}
    if kind == "batch":
        lo = rng.randint(10, 16)
        return {"kind": kind, "jobs": _log_int(rng, 8, 48), "n_lo": lo, "n_hi": lo + rng.randint(2, 4),
                "steps_lo": 10, "steps_hi": rng.randint(20, 60), "mix": rng.randint(1, 1 << 20), "dtype": "c64"}
    if kind == "job":
        fam = rng.choice(["tfim", "heisenberg", "maxcut"])
        n = rng.randint(12, 21)
        return {"kind": kind, "family": fam, "n": _even(n) if fam == "maxcut" else n, "rhs": min(rhs, 4),
                "steps": rng.randint(5, 30), "budget": BUDGET[fam], "dtype": "c64"}
    if kind == "apply":
        fam = rng.choice(["tfim", "heisenberg", "maxcut"])
        n = rng.randint(14, 22)
        return {"kind": kind, "family": fam, "n": _even(n) if fam == "maxcut" else n, "rhs": rhs,
                "budget": BUDGET[fam], "g": rng.randint(0, 8), "dtype": rng.choice(["c64", "c64", "c128"])}
    if kind == "dia":
        return {"kind": kind, "n": rng.randint(10, 16), "rhs": min(rhs, 5), "h": 0.1,
                "dt": math.exp(rng.uniform(math.log(1e-4), math.log(1e-3))), "steps": rng.randint(8, 64),
                "dtype": rng.choice(["c64", "c64", "c128"])}
    if kind == "taylor":
        return {"kind": kind, "n": rng.randint(7, 12), "rhs": min(rhs, 3), "h": 0.1, "budget": rng.randint(256, 768),
                "t": 0.05 + 0.05 * rng.random(), "dtype": rng.choice(["c64", "c128"])}
    fam = rng.choice(["tfim", "heisenberg", "maxcut"])
    n = rng.randint(12, 21)
    return {"kind": kind, "family": fam, "n": _even(n) if fam == "maxcut" else n, "rhs": rhs,
            "dtype": rng.choice(["c64", "c128"])}


# --------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------

def _tdt(case):
    return torch.complex64 if case["dtype"] == "c64" else torch.complex128


def _states(n, rhs, seed, dtype, salt=0):
    """(rhs, 2^n) normalised complex Gaussian states made on the device."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + 17 * n + salt)
    out = torch.empty(rhs, 1 << n, dtype=dtype, device="cuda")
    rdt = torch.float32 if dtype == torch.complex64 else torch.float64
    for r in range(rhs):
        v = torch.randn(1 << n, 2, generator=g, device="cuda", dtype=rdt)
        v /= torch.linalg.vector_norm(v.reshape(-1), dtype=torch.float64).to(rdt)
        out[r] = torch.view_as_complex(v)
    return out


def _ham(family, n, seed, graph=1003):
    """A Hamiltonian of the family: its graph or chain is fixed, its couplings come from the seed."""
    rng = np.random.default_rng(int(seed))
    if family == "tfim":
        return workloads.tfim_chain(n, float(rng.uniform(0.5, 1.5)), float(rng.uniform(0.5, 2.0)))
    if family == "heisenberg":
        return workloads.heisenberg_chain(n, rng.uniform(0.5, 1.5, size=n))
    if family == "maxcut":
        edges = workloads.random_regular_graph(n, 3, np.random.default_rng(graph))
        return workloads.maxcut(n, edges, rng.uniform(0.0, 1.0, size=len(edges)))
    return workloads.tsp_onehot(4, int(seed) % (1 << 31))


def _mix(case, seed):
    """The jobs of a batch: families, sizes, steps and budgets fixed by the mix, couplings by the seed."""
    rng = np.random.default_rng(case["mix"])
    jobs = []
    for k in range(case["jobs"]):
        fam = "tfim" if rng.uniform() < 0.5 else "heisenberg"
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        steps = int(rng.integers(case["steps_lo"], case["steps_hi"] + 1))
        jobs.append((_ham(fam, n, int(seed) * 131 + k), n, steps, int(rng.integers(4, 17))))
    return jobs


def _anneal(case, seed):
    rng = np.random.default_rng(int(seed))
    edges = workloads.random_regular_graph(case["n"], 3, np.random.default_rng(1003))
    cost = workloads.maxcut(case["n"], edges, rng.uniform(0.0, 1.0, size=len(edges)), mixer=0.0)
    n = case["n"]
    labels = [workloads.label_of(n, {i: "X"}) for i in range(n)] + list(cost.labels)
    a = np.concatenate([np.full(n, 0.5), np.zeros(len(cost.labels))])
    b = np.concatenate([np.full(n, -0.5), cost.coeffs])
    return labels, a, b, workloads.midpoint_samples(lambda u: u / 2.0, 2.0, case["steps"])


def _factors(ham, case, t=1.0):
    return hs.hs_build_factors(ham.labels, ham.coeffs, t, max(1, case.get("steps", 20)), case["budget"],
                               case["dtype"], order=case.get("order", 1))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "batch":
        jobs, s["keep"] = [], []
        for k, (ham, n, steps, budget) in enumerate(_mix(case, seed)):
            f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, steps, budget, case["dtype"])
            psi = _states(n, 1, seed, _tdt(case), salt=k)[0]
            jobs.append((f, psi, steps))
        s["psi"] = [j[1] for j in jobs]
        s["batch"] = hs.hs_batch_create(jobs, method=hs.HS_METHOD_REG)
        return s
    if kind in ("dia", "taylor"):
        ham = workloads.tfim_chain(case["n"], 1.0, case["h"])
        s["labels"], s["coeffs"] = ham.labels, ham.coeffs
        s["psi"] = _states(case["n"], case["rhs"], seed, _tdt(case))
        if kind == "dia":
            u = hs.hs_spme(hs.hs_dia_from_terms(ham.labels, ham.coeffs), case["dt"])[0]
            s["u"] = u if case["dtype"] == "c128" else hs.hs_dia_convert(u, "c64")
        else:
            s["psi0"] = s["psi"].clone()
        return s
    s["psi"] = _states(case["n"], case["rhs"], seed, _tdt(case))
    if kind == "anneal":
        labels, a, b, s["drive"] = _anneal(case, seed)
        x, z, n = hs.hs_parse_terms(labels)
        s["f"] = hs.hs_build_factors_td(x, z, a, b, n, 2.0, case["steps"], case["budget"], case["dtype"])
        return s
    ham = _ham(case["family"], case["n"], seed)
    if kind == "evolve":
        s["f"] = _factors(ham, case)
    elif kind == "job":
        s["labels"], s["coeffs"] = ham.labels, ham.coeffs
        s["psi0"], s["out"] = s["psi"].clone(), torch.zeros(case["rhs"], 4, dtype=torch.float64, device="cuda")
    elif kind == "apply":
        s["f"], s["y"] = _factors(ham, case), torch.empty_like(s["psi"])
    else:
        h = hs.hs_dia_from_terms(ham.labels, ham.coeffs)
        s["h"] = h if case["dtype"] == "c128" else hs.hs_dia_convert(h, "c64")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "evolve":
        if case["method"] == "reg":
            hs.hs_evolve_ex(s["f"], s["psi"], case["steps"], method=hs.HS_METHOD_REG)
        else:
            hs.hs_evolve(s["f"], s["psi"], case["steps"])
        return s["psi"]
    if kind == "anneal":
        hs.hs_evolve_td(s["f"], s["psi"], s["drive"], method=hs.HS_METHOD_REG)
        return s["psi"]
    if kind == "batch":
        hs.hs_batch_launch(s["batch"])
        return s["psi"]
    if kind == "job":
        f = hs.hs_build_factors(s["labels"], s["coeffs"], 1.0, case["steps"], case["budget"], case["dtype"])
        s["psi"].copy_(s["psi0"])
        hs.hs_evolve(f, s["psi"], case["steps"])
        for r in range(case["rhs"]):
            hs.hs_inner_device(s["psi0"][r], s["psi"][r], s["out"][r])
        f.close(stream=torch.cuda.current_stream())
        return [s["psi"], s["out"].float()]  # overlaps of single-precision states
    if kind == "apply":
        hs.hs_apply_factor(s["f"], case["g"] % s["f"].n_factors, s["psi"], s["y"])
        return s["y"]
    if kind == "dia":
        hs.hs_dia_evolve(s["u"], s["psi"], case["steps"])
        return s["psi"]
    if kind == "taylor":
        h = hs.hs_dia_from_terms(s["labels"], s["coeffs"])
        r = hs.hs_estimate_timesteps(h, case["t"], case["budget"])
        u, k, _ = hs.hs_spme(h, case["t"] / r)
        if case["dtype"] == "c64":
            u = hs.hs_dia_convert(u, "c64")
        s["psi"].copy_(s["psi0"])
        hs.hs_dia_evolve(u, s["psi"], r)
        return [s["psi"], r, k]
    values, norms = hs.hs_expectation(s["h"], s["psi"])
    return [values, norms]


# --------------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------------

def _n_flips(labels):
    return sum(1 for l in labels if "X" in l or "Y" in l)


def _evolve_flops(labels, n, rhs, steps, order=1):
    """Each flip term two real multiply-adds per amplitude, each step's diagonal terms one complex product."""
    diag = 6 if _n_flips(labels) < len(labels) else 0
    return {1: 1, 2: 2, 4: 10}[order] * steps * (4 * _n_flips(labels) + diag) * rhs * (1 << n)


def _group_masks(labels, budget):
    """x masks of the terms of each budgeted group (next-fit, the offset set capped by the budget)."""
    groups, cur = [], []

    def offsets(xs):
        span = {0}
        for x in xs:
            span |= {v ^ x for v in span}
        offs = set()
        for u in span:
            o = {0}
            for b in range(u.bit_length()):
                if u >> b & 1:
                    o = {v + (1 << b) for v in o} | {v - (1 << b) for v in o}
            offs |= o
        return offs

    for l in labels:
        x = _masks(l)[0]
        if cur and len(offsets(cur + [x])) > budget and offsets(cur + [x]) != offsets(cur):
            groups.append(cur)
            cur = []
        cur = cur + [x]
    groups.append(cur)
    return groups, offsets


def work(case):
    kind, e = case["kind"], 8 if case["dtype"] == "c64" else 16
    if kind == "batch":
        b = f = 0
        for ham, n, steps, _ in _mix(case, 1):
            b += 2 * e * (1 << n)
            f += _evolve_flops(ham.labels, n, 1, steps)
        return {"bytes": b, "flops": f}
    n, rhs = case["n"], case["rhs"]
    state = e * rhs * (1 << n)
    if kind == "evolve":
        labels = _ham(case["family"], n, 1).labels
        return {"bytes": 2 * state, "flops": _evolve_flops(labels, n, rhs, case["steps"], case["order"])}
    if kind == "anneal":
        return {"bytes": 2 * state, "flops": _evolve_flops(_anneal(case, 1)[0], n, rhs, case["steps"])}
    if kind == "job":
        labels = _ham(case["family"], n, 1).labels
        return {"bytes": 2 * state, "flops": _evolve_flops(labels, n, rhs, case["steps"]) + 16 * rhs * (1 << n)}
    if kind == "apply":
        groups, offsets = _group_masks(_ham(case["family"], n, 1).labels, case["budget"])
        offs = offsets(groups[case["g"] % len(groups)])
        stored = sum((1 << n) - abs(d) for d in offs)
        return {"bytes": 2 * state + e * stored, "flops": 8 * rhs * stored}
    if kind == "dia":
        # A truncated exponential of the chain applied step by step: at least the terms of H once per step.
        labels = workloads.tfim_chain(n, 1.0, case["h"]).labels
        return {"bytes": 2 * state, "flops": case["steps"] * (4 * _n_flips(labels) + 6) * rhs * (1 << n)}
    if kind == "taylor":
        labels = workloads.tfim_chain(n, 1.0, case["h"]).labels
        return {"bytes": 2 * state, "flops": 8 * len(labels) * rhs * (1 << n)}
    offs = {0}
    for l in _ham(case["family"], n, 1).labels:
        x, z = _masks(l)
        if x and "Y" not in l:  # a bond's XX and YY cancel on the outer two of its four offsets
            b = [1 << q for q in range(n) if x >> q & 1]
            offs |= {b[0], -b[0]} if len(b) == 1 else {b[1] - b[0], b[0] - b[1]}
    stored = sum((1 << n) - abs(d) for d in offs)
    return {"bytes": state + 16 * rhs + e * stored, "flops": 8 * rhs * stored}


# --------------------------------------------------------------------------------------------
# The same in 64 bits with plain torch
# --------------------------------------------------------------------------------------------

def _masks(label):
    x = z = 0
    n = len(label)
    for k, ch in enumerate(label):
        if ch in "XY":
            x |= 1 << (n - 1 - k)
        if ch in "YZ":
            z |= 1 << (n - 1 - k)
    return x, z


def _view(psi, n, bits):
    """psi (rhs, 2^n) with each of `bits` as an axis of its own: the view and {bit: axis}."""
    shape, axis, top = [psi.shape[0]], {}, n
    for b in sorted(bits, reverse=True):
        shape += [1 << (top - b - 1), 2]
        axis[b] = len(shape) - 1
        top = b
    return psi.view(*shape, 1 << top), axis


def _signs(shape, axes, device):
    """(-1)^(sum of the indices along `axes`), broadcastable to shape."""
    out = torch.ones([1] * len(shape), dtype=torch.float64, device=device)
    for a in axes:
        s = [1] * len(shape)
        s[a] = 2
        out = out * torch.tensor([1.0, -1.0], dtype=torch.float64, device=device).view(s)
    return out


def _pauli(psi, n, x, z):
    """P psi: P|b> = i^popcount(x & z) (-1)^popcount(z & b) |b ^ x>."""
    v, axis = _view(psi, n, [b for b in range(n) if (x | z) >> b & 1])
    if z:
        v = v * _signs(v.shape, [axis[b] for b in range(n) if z >> b & 1], psi.device)
    if x:
        v = torch.flip(v, [axis[b] for b in range(n) if x >> b & 1])
    y = bin(x & z).count("1") % 4
    return (v * (1j ** y) if y else v).reshape(psi.shape)


def _energies(n, terms, device):
    """sum_j c_j (-1)^popcount(z_j & b) over the diagonal terms (c_j, z_j)."""
    e = torch.zeros(1, 1 << n, dtype=torch.float64, device=device)
    for c, z in terms:
        v, axis = _view(e, n, [b for b in range(n) if z >> b & 1])
        v += c * _signs(v.shape, list(axis.values()), device)
    return e


def _step(psi, n, ops, cache):
    """Rotations exp(-i theta P) in order; consecutive diagonal terms as one phase."""
    k = 0
    while k < len(ops):
        x, z, th = ops[k]
        if x == 0:
            run = []
            while k < len(ops) and ops[k][0] == 0:
                run.append((ops[k][2], ops[k][1]))
                k += 1
            key = tuple(run)
            if key not in cache:
                if len(cache) > 4:
                    cache.clear()
                e = _energies(n, run, psi.device)
                cache[key] = torch.complex(torch.cos(e), -torch.sin(e))
            psi.mul_(cache[key])
            continue
        c, s = math.cos(th), math.sin(th)
        if z == 0 and bin(x).count("1") == 1:
            v, axis = _view(psi, n, [x.bit_length() - 1])
            a, b = v.select(2, 0), v.select(2, 1)
            t = a.clone()
            a.mul_(c).add_(b, alpha=-1j * s)
            b.mul_(c).add_(t, alpha=-1j * s)
        else:
            p = _pauli(psi, n, x, z)
            psi.mul_(c).add_(p, alpha=-1j * s)
        k += 1


def _sequence(labels, coeffs, dt, order):
    terms = [(*_masks(l), float(c)) for l, c in zip(labels, coeffs)]

    def strang(h):
        half = [(x, z, c * (0.5 * h)) for x, z, c in terms]
        return half + half[::-1]

    if order == 1:
        return [(x, z, c * dt) for x, z, c in terms]
    if order == 2:
        return strang(dt)
    p = 1.0 / (4.0 - 4.0 ** (1.0 / 3.0))
    return strang(p * dt) * 2 + strang((1.0 - 4.0 * p) * dt) + strang(p * dt) * 2


def _apply_h(psi, n, terms, diag):
    out = psi * diag
    for x, z, c in terms:
        out += c * _pauli(psi, n, x, z)
    return out


def _split(labels, coeffs, n, device):
    flips = [(*_masks(l), float(c)) for l, c in zip(labels, coeffs)]
    diag = _energies(n, [(c, z) for x, z, c in flips if not x], device)
    return [t for t in flips if t[0]], diag


def _seconds(case):
    """About how long exact() takes: a term costs some launches or some passes over the states."""
    kind = case["kind"]
    if kind == "batch":
        return sum(steps * (_n_flips(h.labels) + 1) * (6e-5 + 16 * 8 * (1 << n) / 3e12) for h, n, steps, _ in _mix(case, 1))
    n, rhs = case["n"], case["rhs"]
    one = 6e-5 + 16 * rhs * (1 << n) * 6 / 3e12
    if kind in ("evolve", "anneal", "job"):
        labels = _anneal(case, 1)[0] if kind == "anneal" else _ham(case["family"], n, 1).labels
        return case["steps"] * {1: 1, 2: 2, 4: 10}[case.get("order", 1)] * (_n_flips(labels) + 2) * one
    if kind == "taylor":
        return 10 * 60 * n * one  # one long exponential
    if kind == "dia":
        return case["steps"] * 8 * n * one
    return 1.0


def exact(case, seed):
    if _seconds(case) > 16:
        return None
    kind = case["kind"]
    if kind == "batch":
        out = []
        for k, (ham, n, steps, _) in enumerate(_mix(case, seed)):
            psi = _states(n, 1, seed, _tdt(case), salt=k).to(torch.complex128)
            ops, cache = _sequence(ham.labels, ham.coeffs, 1.0 / steps, 1), {}
            for _ in range(steps):
                _step(psi, n, ops, cache)
            out.append(psi[0])
        return out
    n = case["n"]
    psi = _states(n, case["rhs"], seed, _tdt(case)).to(torch.complex128)
    if kind == "anneal":
        labels, a, b, drive = _anneal(case, seed)
        for f in drive:
            _step(psi, n, _sequence(labels, a + f * b, 2.0 / case["steps"], 1), {})
        return psi
    if kind in ("evolve", "job"):
        ham = _ham(case["family"], n, seed)
        psi0 = psi.clone() if kind == "job" else None
        ops, cache = _sequence(ham.labels, ham.coeffs, 1.0 / case["steps"], case.get("order", 1)), {}
        for _ in range(case["steps"]):
            _step(psi, n, ops, cache)
        if kind == "evolve":
            return psi
        ip = (psi0.conj() * psi).sum(1)
        return [psi, torch.stack([ip.real, ip.imag, psi0.abs().square().sum(1), psi.abs().square().sum(1)], 1)]
    if kind == "apply":
        ham = _ham(case["family"], n, seed)
        groups, _ = _group_masks(ham.labels, case["budget"])
        g = case["g"] % len(groups)
        k0 = sum(len(v) for v in groups[:g])
        _step(psi, n, _sequence(ham.labels, ham.coeffs, 1.0 / max(1, case.get("steps", 20)), 1)[k0:k0 + len(groups[g])], {})
        return psi
    if kind == "expect":
        ham = _ham(case["family"], n, seed)
        flips, diag = _split(ham.labels, ham.coeffs, n, psi.device)
        v = (psi.conj() * _apply_h(psi, n, flips, diag)).sum(1)
        return [v.cpu().numpy(), psi.abs().square().sum(1).cpu().numpy()]
    # The exponential of the chain by its Taylor series on the states, in steps short enough to converge.
    flips, diag = _split(workloads.tfim_chain(n, 1.0, case["h"]).labels, workloads.tfim_chain(n, 1.0, case["h"]).coeffs,
                         n, psi.device)
    total = case["dt"] * case["steps"] if kind == "dia" else case["t"]
    m = max(1, math.ceil(total * 2 * n))
    for _ in range(m):
        term = psi.clone()
        for k in range(1, 26):
            term = _apply_h(term, n, flips, diag) * (-1j * total / m / k)
            psi = psi + term
    return psi if kind == "dia" else [psi, None, None]
