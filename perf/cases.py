"""What the engine's users have it do, as measurable cases.

A case is one call through the package's public entry points on a seeded
d-regular Max-Cut graph: the QAOA objective <C> of all edge networks (on
device buffers, on host values, or as an autograd step), one edge network
alone, or the full state vector.  The sizes are those of the workloads,
tests and benchmark of this repository (n = 12 to 100 vertices, degree 3 to
7, depth 1 to 3); `draw` spreads over the same ranges.

Single-precision runs (complex64 and split BF16) return their values as
float32, the precision they are computed in; complex128 runs return float64.
The angles are drawn from the seed; the graph belongs to the case.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1709_03636_gb300 as qtc

FULL = dict(call="device", n=0, d=0, p=1, graph=0, dtype="c64", diag=True, cone=True,
            ordering="lg", restarts=8, grad=False, noise=0.0, per_edge=False)


def _case(name, **fields):
    return {"name": name, **FULL, **fields}


def listed():
    return [
        # the smallest objective, to full precision, values in and out on the host: what
        # an optimiser running on the CPU calls thousands of times
        _case("p1_n12_host_c128", call="host", n=12, d=3, dtype="c128", diag=False,
              ordering="stoch", grad=True),
        # the everyday p = 1 objective and gradient from the host
        _case("p1_n50_host", call="host", n=50, d=3, grad=True),
        # the same graph size with depolarising noise after the mixer, device buffers
        _case("p1_n51_noisy", n=51, d=4, grad=True, noise=0.03),
        # a p = 2 optimisation step: forward and backward through autograd
        _case("p2_n100_step", call="autograd", n=100, d=5, p=2, grad=True),
        # the paper's dense rank-4 gate form: tensor cores forward, FP32 with the gradient
        _case("p2_n100_dense_bf16", n=100, d=5, p=2, dtype="split_bf16", diag=False),
        _case("p2_n100_dense_grad", n=100, d=5, p=2, diag=False, grad=True),
        # the headline: depth 3, value and gradient of 120 large networks
        _case("p3_n60_grad", n=60, d=4, p=3, restarts=64, grad=True),
        # one large edge network alone: little parallelism between networks
        _case("p3_n60_edge", call="edge", n=60, d=4, p=3, restarts=64, grad=True),
        # un-reduced networks, as in the crossover study: the largest intermediates ...
        _case("p1_n26_full", n=26, d=7, cone=False),
        # ... and in double precision with the gradient
        _case("p1_n20_full_c128", n=20, d=7, cone=False, dtype="c128", grad=True),
        # the state vector beside it: beyond L2, and depth 3 within L2 with per-edge values
        _case("sv_n26", call="state", n=26, d=7),
        _case("sv_n21_p3_edges", call="state", n=21, d=6, p=3, per_edge=True),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["p1", "p1", "p2", "dense", "p3", "edge", "full", "state", "state"])
    c = dict(FULL, graph=rng.randrange(1, 1 << 20))
    if kind == "p1":
        c.update(call=rng.choice(["host", "device", "autograd"]), n=spread(9, 200),
                 d=rng.randint(3, 6), dtype=rng.choice(["c64", "c64", "c128"]),
                 diag=rng.random() < 0.7, ordering=rng.choice(["lg", "lg", "stoch"]),
                 grad=rng.random() < 0.6, noise=rng.choice([0.0, 0.0, 0.02, 0.1]))
        if c["noise"]:
            c.update(diag=True, ordering="lg", d=min(c["d"], 4))
    elif kind == "p2":
        c.update(call=rng.choice(["host", "device", "autograd"]), n=spread(30, 120),
                 d=rng.randint(3, 5), p=2, grad=rng.random() < 0.7)
    elif kind == "dense":
        c.update(n=spread(20, 100), d=rng.randint(3, 5), p=2, diag=False,
                 dtype=rng.choice(["split_bf16", "c64"]), grad=rng.random() < 0.5)
    elif kind == "p3":
        c.update(n=spread(24, 60), d=rng.choice([3, 3, 4]), p=3, restarts=rng.choice([8, 64]),
                 grad=rng.random() < 0.7)
    elif kind == "edge":
        c.update(call="edge", n=spread(30, 60), d=rng.choice([3, 4]), p=3, restarts=64,
                 grad=rng.random() < 0.5)
    elif kind == "full":
        c.update(n=rng.randint(14, 23), d=rng.randint(3, 6), cone=False,
                 dtype=rng.choice(["c64", "c64", "c128"]), grad=rng.random() < 0.5)
    else:
        c.update(call="state", n=rng.randint(10, 26), d=rng.randint(3, 7), p=rng.randint(1, 3),
                 dtype=rng.choice(["c64", "c64", "c128"]), per_edge=rng.random() < 0.4)
    if c["call"] == "autograd":
        c["grad"] = True
    if c["n"] * c["d"] % 2:
        c["n"] += 1
    return c


def _graph(case):
    """A connected random d-regular graph: random stub pairing, repaired by edge swaps."""
    n, d = case["n"], case["d"]
    rng = random.Random(1000003 * case["graph"] + 1009 * n + d)
    while True:
        stubs = [v for v in range(n) for _ in range(d)]
        rng.shuffle(stubs)
        pairs = [tuple(sorted(stubs[i:i + 2])) for i in range(0, n * d, 2)]
        for _ in range(200 * n * d):
            bad = [i for i, e in enumerate(pairs) if e[0] == e[1] or pairs.count(e) > 1]
            if not bad:
                break
            i, j = bad[0], rng.randrange(len(pairs))
            (a, b), (u, v) = pairs[i], pairs[j]
            pairs[i], pairs[j] = tuple(sorted((a, u))), tuple(sorted((b, v)))
        else:
            continue
        reach, todo = {0}, [0]
        while todo:
            a = todo.pop()
            for e in pairs:
                if a in e:
                    b = e[0] + e[1] - a
                    if b not in reach:
                        reach.add(b)
                        todo.append(b)
        if len(reach) == n:
            return sorted(pairs)


def _angles(case, seed):
    rng = random.Random(seed)
    g = [rng.uniform(0.0, math.pi) for _ in range(case["p"])]
    b = [rng.uniform(0.0, math.pi / 2) for _ in range(case["p"])]
    if case["call"] == "autograd" and case["dtype"] != "c128":
        g, b = ([float(np.float32(x)) for x in v] for v in (g, b))  # float32 parameters
    return g, b


def _real(case):
    return torch.float64 if case["dtype"] == "c128" else torch.float32


def _circuit(case):
    noise = ("depolarize", case["noise"]) if case["noise"] else None
    return qtc.Circuit.qaoa(case["n"], _graph(case), case["p"], noise=noise)


def _arena(case):
    if case["call"] == "state":
        return (16 << case["n"]) + (64 << 20)
    return 12 << 30 if case["p"] == 3 or not case["cone"] else 1 << 30


def prepare(case, seed):
    g, b = _angles(case, seed)
    circuit = _circuit(case)
    engine = qtc.Engine(0, arena_bytes=_arena(case))
    s = dict(case=case, circuit=circuit, engine=engine, g=g, b=b)
    m = len(circuit.edges)
    if case["call"] == "state":
        s["params"] = torch.tensor(g + b, dtype=torch.float64, device="cuda")
        s["out"] = torch.zeros(1 + m, dtype=torch.float64, device="cuda")
        return s
    if case["call"] == "edge":
        net = qtc.Network(circuit, edge=circuit.edges[m // 2])
        s["plan"] = qtc.Plan(net, case["ordering"], restarts=case["restarts"])
        return s
    s["batch"] = qtc.Batch(circuit, lightcone=case["cone"], diag=case["diag"],
                           ordering=case["ordering"], restarts=case["restarts"])
    s["batch"].prepare(engine, case["dtype"], want_grad=case["grad"])
    if case["call"] == "autograd":
        s["params"] = torch.tensor(g + b, dtype=_real(case), device="cuda", requires_grad=True)
    elif case["call"] == "device":
        s["params"] = torch.tensor(g + b, dtype=torch.float64, device="cuda")
        s["out"] = torch.zeros(2 + 2 * case["p"] + m, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case, engine = s["case"], s["engine"]
    dtype, grad, P = case["dtype"], case["grad"], 2 * case["p"]
    if case["call"] == "state":
        out = qtc.statevector_expectation_device(engine, s["circuit"], s["params"], s["out"],
                                                 dtype, per_edge=case["per_edge"])
        out = out.to(_real(case))
        return {"C": out[:1], "zz": out[1:]} if case["per_edge"] else {"C": out[:1]}
    if case["call"] == "edge":
        got = qtc.contract(engine, s["plan"], s["g"] + s["b"], dtype, want_grad=grad)
        value, slopes = got if grad else (got, [])
        real = np.float64 if dtype == "c128" else np.float32
        r = {"zz": np.array([value.real], dtype=real)}
        return dict(r, grad=np.array([v.real for v in slopes], dtype=real)) if grad else r
    if case["call"] == "autograd":
        x = s["params"]
        x.grad = None
        c = qtc.QAOAExpectation.apply(x, engine, s["batch"], dtype)
        c.backward()
        return {"C": c.detach(), "grad": x.grad}
    if case["call"] == "host":
        c, zz, slopes = qtc.qaoa_expectation(engine, s["batch"], s["g"], s["b"], dtype,
                                             want_grad=grad)
        real = np.float64 if dtype == "c128" else np.float32
        r = {"C": np.array([c], dtype=real), "zz": np.array(zz, dtype=real)}
        return dict(r, grad=np.array(slopes, dtype=real)) if grad else r
    out = qtc.qaoa_expectation_device(engine, s["batch"], s["params"], s["out"], dtype,
                                      want_grad=grad).to(_real(case))
    r = {"C": out[:1], "zz": out[1 + P:-1]}
    return dict(r, grad=out[1:1 + P]) if grad else r


def work(case):
    """Angles in, values out; the arithmetic of the state vector's layers, or
    of the contraction plans that the case names (8 per complex multiply-add)."""
    edges, p, n = _graph(case), case["p"], case["n"]
    nbytes = 8 * (2 * p + 1 + (2 * p if case["grad"] else 0) + len(edges))
    if case["call"] == "state":
        # per layer a phase product (6) and n two-term rotations (4 each) per amplitude,
        # then |psi|^2 weighted (5; per edge 1)
        flops = (p * (6 + 4 * n) + 5 + (len(edges) if case["per_edge"] else 0)) * 2.0 ** n
        return {"bytes": nbytes, "flops": flops}
    only = [edges[len(edges) // 2]] if case["call"] == "edge" else None
    st = qtc.Batch(_circuit(case), only, lightcone=case["cone"], diag=case["diag"],
                   ordering=case["ordering"], restarts=case["restarts"]).stats()
    return {"bytes": nbytes,
            "flops": 8.0 * (st["cmacs"] + (st["grad_cmacs"] if case["grad"] else 0))}


# ---- the same values in 64 bits, from torch alone ------------------------------


def _zz_gate(g):
    z = torch.tensor([[1.0, -1.0], [-1.0, 1.0]], dtype=torch.float64, device=g.device)
    return torch.complex(torch.cos(g * z / 2), -torch.sin(g * z / 2))


def _rx_gate(b):
    c, s, o = torch.cos(b), torch.sin(b), torch.zeros_like(b)
    return torch.stack([torch.complex(c, o), torch.complex(o, -s), torch.complex(o, -s),
                        torch.complex(c, o)]).reshape(2, 2)


def _edge_factors(edges, near, edge, zz, rx):
    """(tensor, labels) of <Z_u Z_v> for one edge: the gates in its reverse
    light cone, ket and bra, wires of other qubits joined."""
    p = len(zz)
    balls = [set(edge)]
    for _ in range(p):
        balls.append(balls[-1] | {b for a in balls[-1] for b in near[a]})
    count, out, ends = 0, [], []
    half = torch.full((2,), math.sqrt(0.5), dtype=torch.complex128, device=zz[0].device)
    for side in (0, 1):
        at = {}
        for q in balls[p]:
            at[q], count = count, count + 1
            out.append((half, [at[q]]))
        for k in range(p):
            core = balls[p - 1 - k]
            zk, rk = (zz[k], rx[k]) if side == 0 else (zz[k].conj(), rx[k].conj())
            out += [(zk, [at[a], at[b]]) for a, b in edges if a in core or b in core]
            for q in core:
                out.append((rk, [count, at[q]]))
                at[q], count = count, count + 1
        ends.append(at)
    z = torch.tensor([1.0, -1.0], dtype=torch.complex128, device=half.device)
    joined = {ends[1][q]: ends[0][q] for q in balls[p]}
    out = [(t, [joined.get(x, x) for x in ls]) for t, ls in out]
    return out + [(z, [ends[0][q]]) for q in edge]


def _fill_order(factors):
    """Elimination order by least fill, on neighbour sets held as bit masks."""
    nb = {}
    for _, ls in factors:
        mask = sum(1 << x for x in ls)
        for x in ls:
            nb[x] = nb.get(x, 0) | mask
    nb = {x: m & ~(1 << x) for x, m in nb.items()}

    def bits(m):
        while m:
            low = m & -m
            yield low.bit_length() - 1
            m ^= low

    cost, stale, order = {}, set(nb), []
    while nb:
        for x in stale:
            if x in nb:
                m = nb[x]
                cost[x] = (sum((m & ~nb[y]).bit_count() - 1 for y in bits(m)), m.bit_count(), x)
        x = min(nb, key=cost.__getitem__)
        m = nb.pop(x)
        stale = set(bits(m))
        for y in bits(m):
            nb[y] = (nb[y] | m) & ~((1 << x) | (1 << y))
        for y in list(stale):
            stale.update(bits(nb[y]))
        order.append(x)
    return order


def _contract(factors):
    factors = list(factors)
    for x in _fill_order(factors):
        hold = sorted((f for f in factors if x in f[1]), key=lambda f: f[0].dim())
        factors = [f for f in factors if x not in f[1]]
        keep = sorted({y for _, ls in hold for y in ls} - {x})
        place = {y: i for i, y in enumerate(keep + [x])}
        args = [a for t, ls in hold for a in (t, [place[y] for y in ls])]
        factors.append((torch.einsum(*args, [place[y] for y in keep]), keep))
    value = factors[0][0]
    for t, _ in factors[1:]:
        value = value * t
    return value.real


def _exact_networks(case, seed):
    edges = _graph(case)
    near = {}
    for a, b in edges:
        near.setdefault(a, []).append(b)
        near.setdefault(b, []).append(a)
    g, b = _angles(case, seed)
    theta = torch.tensor(g + b, dtype=torch.float64, device="cuda", requires_grad=True)
    # depolarising after the only mixer damps Z on each of the two qubits
    damp = (1 - 4 * case["noise"] / 3) ** 2
    zz_all, slopes = [], torch.zeros_like(theta)
    for e in [edges[len(edges) // 2]] if case["call"] == "edge" else edges:
        with torch.set_grad_enabled(case["grad"]):
            zz = [_zz_gate(theta[k]) for k in range(case["p"])]
            rx = [_rx_gate(theta[case["p"] + k]) for k in range(case["p"])]
            v = damp * _contract(_edge_factors(edges, near, e, zz, rx))
        zz_all.append(v.detach())
        if case["grad"]:
            slopes += torch.autograd.grad(v, theta)[0]
    return torch.stack(zz_all), slopes


def _exact_state(case, seed):
    edges, n = _graph(case), case["n"]
    g, b = _angles(case, seed)
    x = torch.arange(1 << n, device="cuda")
    cut = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
    for a, c in edges:
        cut += ((x >> a) ^ (x >> c)) & 1
    psi = torch.full((1 << n,), 2.0 ** (-n / 2), dtype=torch.complex128, device="cuda")
    for k in range(case["p"]):
        angle = -g[k] * (len(edges) - 2 * cut) / 2
        psi *= torch.complex(torch.cos(angle), torch.sin(angle))
        co, si = math.cos(b[k]), math.sin(b[k])
        for q in range(n):
            v = psi.view(-1, 2, 1 << q)
            psi = (co * v - 1j * si * v.flip(1)).reshape(-1)
    prob = psi.real ** 2 + psi.imag ** 2
    r = {"C": (prob * cut).sum().reshape(1)}
    if case["per_edge"]:
        r["zz"] = torch.stack([(prob * (1 - 2 * (((x >> a) ^ (x >> c)) & 1))).sum()
                               for a, c in edges])
    return r


def exact(case, seed):
    if case["call"] == "state":
        return _exact_state(case, seed)
    zz, slopes = _exact_networks(case, seed)
    if case["call"] == "edge":
        return {"zz": zz, "grad": slopes} if case["grad"] else {"zz": zz}
    c = ((1 - zz) / 2).sum()
    if case["call"] == "autograd":
        return {"C": c, "grad": -slopes / 2}
    r = {"C": c.reshape(1), "zz": zz}
    return dict(r, grad=-slopes / 2) if case["grad"] else r
