"""The work a user has this library do, as timed cases over its public entry points.

Every kind of call the library offers for a solve is here, over the sizes of its own
configurations, tests and benchmark: one instance from the smallest (a few microseconds a
generation) to a population of hundreds of millions of qubits, both rotation rules, items
that do and do not fit a byte, the convergence stop, many instances in one call, the solve
server, one generation at a time on the caller's own device buffers, and one block of rows of
a sharded population.

A pass starts every solve at generation 0, so it can be repeated on the same state.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_30862_gb300 import qieo as Q
from paper_2609_30862_gb300 import workload as W


def listed():
    return [
        # The smallest population a served or batched solve has, for one step of generations:
        # launches, the reset and the read of the best record are most of the call.
        {"name": "tiny_solve", "kind": "solve", "np": 32, "ng": 50, "gens": 25},
        # The smallest named workload: 64 chromosomes, 100 items, 500 generations.
        {"name": "small_solve", "kind": "solve", "np": 64, "ng": 100, "gens": 500},
        # An ordinary solve of uneven size under the rule that only moves qubits whose allele
        # differs from the elite's, with a finer angle step and a heavier penalty.
        {"name": "ragged_solve_r2", "kind": "solve", "np": 500, "ng": 5003, "gens": 300, "rule": 1, "D": 200,
         "lam": 3},
        # The named workload whose population fits on chip: 1,024 x 10,000, 1,000 generations.
        {"name": "onchip_solve", "kind": "solve", "np": 1024, "ng": 10000, "gens": 1000},
        # The named workload that streams from device memory: 4,096 x 100,000, 200 generations.
        {"name": "streamed_solve", "kind": "solve", "np": 4096, "ng": 100000, "gens": 200},
        # The first generations of a large population, as the (Np, Ng) sweep times them: every
        # qubit is still drawn. Ragged in both sizes.
        {"name": "spread_population", "kind": "solve", "np": 6001, "ng": 70001, "gens": 24},
        # Items that do not fit a byte (prices, byte sizes): the 64-bit item sums.
        {"name": "wide_items", "kind": "solve", "np": 777, "ng": 20011, "gens": 60, "items": "wide"},
        # Solve until the elite's fitness has been stable (Sec. IV), at most 400 generations.
        {"name": "converge_stop", "kind": "solve", "np": 256, "ng": 2003, "gens": 400, "converge": True},
        # Independent instances of uneven sizes in one call (parameter studies, portfolios).
        {"name": "batch", "kind": "batch", "count": 96, "gens": 200, "sizes": 1},
        # The same kind of requests through the solve server: submitted, admitted, polled back.
        {"name": "server", "kind": "serve", "count": 64, "gens": 100, "sizes": 2},
        # Single generations on buffers the caller owns (a loop that may not allocate).
        {"name": "caller_buffers", "kind": "noalloc", "np": 512, "ng": 10007, "gens": 4},
        # One rank's block of rows of a population sharded over devices: observe, find the
        # elite, rotate toward the row the ranks agreed on.
        {"name": "row_block", "kind": "rows", "np": 1500, "ng": 20000, "gens": 10, "row0": 1500},
    ]


def _log_uniform(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["wide", "converge", "batch", "serve", "noalloc", "rows"])
    if kind == "batch":
        return {"kind": "batch", "count": _log_uniform(rng, 8, 256), "gens": _log_uniform(rng, 20, 300),
                "sizes": rng.randrange(3, 1 << 20)}
    if kind == "serve":
        return {"kind": "serve", "count": _log_uniform(rng, 8, 128), "gens": _log_uniform(rng, 20, 150),
                "sizes": rng.randrange(3, 1 << 20)}
    if kind == "noalloc":
        n = _log_uniform(rng, 32, 4096)
        return {"kind": "noalloc", "np": n, "ng": _log_uniform(rng, 50, min(50000, 30_000_000 // n)),
                "gens": rng.randint(1, 6), "rule": rng.randint(0, 1)}
    if kind == "rows":
        n = _log_uniform(rng, 32, 4096)
        return {"kind": "rows", "np": n, "ng": _log_uniform(rng, 50, min(100000, 100_000_000 // n)),
                "gens": rng.randint(3, 12), "row0": rng.randrange(0, 10000), "rule": rng.randint(0, 1)}
    c = {"kind": "solve"}
    n = _log_uniform(rng, 32, 16384)
    if kind == "wide":      # the 64-bit sums cost more a gene
        g = _log_uniform(rng, 50, min(50000, 60_000_000 // n))
        most = 2_000_000_000
        c["items"] = "wide"
    elif kind == "converge":
        g = _log_uniform(rng, 50, min(50000, 60_000_000 // n))
        most = 8_000_000_000
        c["converge"] = True
    else:
        g = _log_uniform(rng, 50, min(200000, 600_000_000 // n))
        most = 16_000_000_000
    c.update(np=n, ng=g, gens=_log_uniform(rng, 10, max(10, min(1000, most // (n * g)))))
    c["rule"] = rng.choice([0, 0, 1])
    c["D"] = rng.choice([100, 100, 100, 40, 200])
    c["lam"] = rng.choice([1, 1, 7])
    return c


def _problem(case, seed):
    if case.get("items") != "wide":
        return W.knapsack(case["ng"], seed)
    # weights up to 5,000 and values loosely tied to them: neither fits a byte
    r = np.random.RandomState(seed % (1 << 32))
    w = r.randint(1, 5001, case["ng"]).astype(np.int32)
    v = (w // 2 + r.randint(1, 5001, case["ng"])).astype(np.int32)
    return W.custom_problem(w, v, int(w.astype(np.int64).sum()) // 2)


def _manifest(case, seed):
    return W.batch_manifest(case["count"], manifest_seed=1000 + case["sizes"], first_seed=1 + seed % (1 << 30))


def _instance(case, problem, seed, row0=None):
    flags = Q.QIEO_FLAG_CONVERGE if case.get("converge") else 0
    return Q.Instance(problem, case["np"], seed=seed, inst=0, D=case.get("D", 100), lam=case.get("lam", 1),
                      rule=case.get("rule", 0), flags=flags, row0=row0)


def _mid_run_indices(case, seed):
    """Angle indices of a population part of the way to its bounds: some qubits at 0 and
    pi/2, the rest between."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.randn((case["np"], case["ng"]), generator=g, device="cuda") * 16.0
    return k.round().clamp(-25, 25).to(torch.int16).contiguous()


def prepare(case, seed):
    Q.load()
    seed = int(seed)
    kind = case["kind"]
    s = {"case": case, "kind": kind, "seed": seed}
    if kind == "batch":
        s["members"] = [Q.Instance(W.knapsack(m.ng, m.seed), m.np_, seed=m.seed, inst=m.seed)
                        for m in _manifest(case, seed)]
        s["batch"] = Q.Batch(s["members"])
        return s
    if kind == "serve":
        s["requests"] = [(W.knapsack(m.ng, m.seed), m) for m in _manifest(case, seed)]
        s["server"] = Q.Server(memory_bytes=4 << 30, gens_per_step=25)
        return s
    problem = _problem(case, seed)
    s["problem"] = problem
    if kind == "noalloc":
        n, ng = case["np"], case["ng"]
        dev = torch.device("cuda")
        s["w"] = torch.from_numpy(problem.weights).to(dev)
        s["v"] = torch.from_numpy(problem.values).to(dev)
        s["k0"] = _mid_run_indices(case, seed)
        s["k"] = torch.empty_like(s["k0"])
        s["x"] = torch.zeros((n, ng), dtype=torch.uint8, device=dev)
        s["f"] = torch.zeros(n, dtype=torch.int64, device=dev)
        s["e"] = torch.zeros(1, dtype=torch.int32, device=dev)
        p = Q.qieo_default_params()
        p.np, p.seed, p.rotate_rule = n, seed & 0xFFFFFFFF, case.get("rule", 0)
        s["params"] = p
        return s
    s["inst"] = _instance(case, problem, seed, row0=case.get("row0"))
    return s


def _records(inst, gens):
    """The solve's result and its course: the best record, the elite of every generation and
    the last population's fitness (and the angle indices, where reading them is a small part
    of the call)."""
    bits, f, g, c = inst.best()
    e, fe = inst.history(0, gens)
    out = {"best_alleles": bits, "best": np.array([f, g, c], dtype=np.int64), "elite": e, "elite_fitness": fe,
           "fitness": inst.fitness()}
    if inst.np_ * inst.ng <= 1 << 14:
        out["state"] = inst.state()[0]
    return out


def _run_solve(s):
    inst, case = s["inst"], s["case"]
    inst.reset()
    if case.get("converge"):
        inst.run(case["gens"])
        stopped, stable = inst.convergence()
        bits, f, g, c = inst.best()
        return {"best_alleles": bits, "best": np.array([f, g, c], dtype=np.int64),
                "stopped": np.array([stopped, stable], dtype=np.int64), "fitness": inst.fitness()}
    inst.run(case["gens"])
    return _records(inst, case["gens"])


def _run_batch(s):
    for m in s["members"]:
        m.reset()
    s["batch"].run(s["case"]["gens"])
    best = [m.best() for m in s["members"]]
    return {"alleles": np.concatenate([b[0] for b in best]),
            "best": np.array([b[1:] for b in best], dtype=np.int64)}


def _run_serve(s):
    srv, gens = s["server"], s["case"]["gens"]
    ids = [srv.submit(p, m.np_, gens, seed=m.seed, inst=m.seed) for p, m in s["requests"]]
    bits, best = [], []
    for rid in ids:
        res, x = srv.poll(rid, wait_ms=60000)
        bits.append(x)
        best.append((res.state, res.fitness, res.generation, res.chromosome))
    return {"alleles": np.concatenate(bits), "best": np.array(best, dtype=np.int64)}


def _run_noalloc(s):
    s["k"].copy_(s["k0"])
    p, case = s["params"], s["case"]
    p.stream = torch.cuda.current_stream().cuda_stream
    for t in range(case["gens"]):
        Q.qieo_generation_noalloc(s["w"].data_ptr(), s["v"].data_ptr(), case["ng"], s["problem"].capacity, p, t,
                                  s["k"].data_ptr(), s["x"].data_ptr(), s["f"].data_ptr(), s["e"].data_ptr())
    return {"k": s["k"], "x": s["x"], "fitness": s["f"], "elite": s["e"]}


def _run_rows(s):
    inst, row0 = s["inst"], s["case"]["row0"]
    inst.reset()
    found = []
    for t in range(s["case"]["gens"]):
        f, c = inst.rows_observe(t)
        elite = inst.allele_row(c - row0)
        inst.rows_rotate(elite)
        found.append((f, c))
    return {"found": np.array(found, dtype=np.int64), "elite": elite, "fitness": inst.fitness()}


def run(state):
    return {"solve": _run_solve, "batch": _run_batch, "serve": _run_serve, "noalloc": _run_noalloc,
            "rows": _run_rows}[state["kind"]](state)


def work(case):
    """Bytes: the items and, where the call is given or leaves a population, the angle indices
    and alleles, each once. Operations: per qubit and generation a quarter of a Philox4x32-10
    call (10 rounds of 2 multiplies and 4 xors), the rotation (3), the compare and two sums;
    qubits fixed at a bound need none of it, which this figure does not count."""
    per_gene = 21.0
    if case["kind"] in ("batch", "serve"):
        m = _manifest(case, 1)
        genes, cells, rows = sum(x.ng for x in m), sum(x.ng * x.np_ for x in m), sum(x.np_ for x in m)
    else:
        genes, rows = case["ng"], case["np"]
        cells = genes * rows
    state = cells * (5.0 if case["kind"] == "noalloc" else 2.125)
    return {"bytes": 8.0 * genes + state + 8.0 * rows, "flops": per_gene * cells * case["gens"]}


# ---------------------------------------------------------------------------------------
# The same results from the definition, in 64-bit integers.
# ---------------------------------------------------------------------------------------
def _thresholds(D):
    K = D // 4
    # T[n] = round(sin^2(n pi / D) 2^32) in decimal arithmetic with room to spare
    import decimal
    decimal.getcontext().prec = 50
    Dec = decimal.Decimal
    pi = Dec("3.14159265358979323846264338327950288419716939937510")

    def cos(x):
        term, total, n = Dec(1), Dec(1), 0
        while abs(term) > Dec(10) ** -45:
            n += 2
            term = -term * x * x / (n * (n - 1))
            total += term
        return total
    T = [0] * (2 * K + 1)
    for n in range(K + 1):
        T[n] = int((Dec(2) ** 31 * (1 - cos(2 * pi * n / D))).to_integral_value(decimal.ROUND_HALF_UP))
    T[0], T[K] = 0, 1 << 31
    for n in range(K + 1, 2 * K + 1):
        T[n] = (1 << 32) - T[2 * K - n]
    return T


def _draws(rows, ng, t, seed, inst, dev):
    """Philox4x32-10 words of genes 0 .. ng - 1 of the given rows at generation t."""
    m32 = 0xFFFFFFFF
    c0 = torch.arange((ng + 3) // 4, device=dev, dtype=torch.int64)[None, :].expand(len(rows), -1).contiguous()
    c1 = rows[:, None].expand_as(c0).contiguous()
    c2 = torch.full_like(c0, t)
    c3 = torch.zeros_like(c0)
    k0, k1 = seed & m32, inst & m32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57     # 64-bit products, wrapped into int64
        c0, c1, c2, c3 = (((p1 >> 32) & m32) ^ c1 ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c3 ^ k1, p0 & m32)
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return torch.stack([c0, c1, c2, c3], dim=2).reshape(len(rows), -1)[:, :ng]


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind in ("batch", "serve") or case["gens"] * (case["np"] * case["ng"] + 2_000_000) > 3_000_000_000:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    n, ng, D, lam = case["np"], case["ng"], case.get("D", 100), case.get("lam", 1)
    rule, K, problem = case.get("rule", 0), D // 4, _problem(case, seed)
    w = torch.from_numpy(problem.weights).to(dev).long()
    v = torch.from_numpy(problem.values).to(dev).long()
    T = torch.tensor(_thresholds(D), device=dev, dtype=torch.int64)
    rows = torch.arange(n, device=dev, dtype=torch.int64) + case.get("row0", 0)
    k = _mid_run_indices(case, seed).long() if kind == "noalloc" else torch.zeros((n, ng), device=dev, dtype=torch.int64)
    hist_e, hist_f, best, stable, stopped = [], [], None, 0, 0
    for t in range(case["gens"]):
        x = (_draws(rows, ng, t, seed, 0, dev) < T[k + K]).long()
        sw, sv = (x * w).sum(1), (x * v).sum(1)
        f = torch.where(sw <= problem.capacity, sv, -lam * (sw - problem.capacity))
        fe = int(f.max())
        e = int((f == fe).nonzero()[0, 0])
        if best is None or fe > best[0]:
            best = (fe, t, e, x[e].clone())
        stable = stable + 1 if hist_f and hist_f[-1] == fe else 1
        hist_e.append(e)
        hist_f.append(fe)
        step = (2 * x[e] - 1)[None, :].expand_as(k)
        if rule == 1:
            step = torch.where(x == x[e][None, :], torch.zeros_like(step), step)
        k = (k + step).clamp(-K, K)
        if case.get("converge") and stable >= 20:
            stopped = 1
            break
    fit = f.cpu().numpy()
    if kind == "noalloc":
        return {"k": k.to(torch.int16), "x": x.to(torch.uint8), "fitness": f,
                "elite": torch.tensor([e], dtype=torch.int32)}
    if kind == "rows":
        found = np.array([(a, b + case["row0"]) for a, b in zip(hist_f, hist_e)], dtype=np.int64)
        return {"found": found, "elite": x[e].to(torch.uint8).cpu().numpy(), "fitness": fit}
    bits = best[3].to(torch.uint8).cpu().numpy()
    rec = np.array(best[:3], dtype=np.int64)
    if case.get("converge"):
        return {"best_alleles": bits, "best": rec, "stopped": np.array([stopped, stable], dtype=np.int64),
                "fitness": fit}
    out = {"best_alleles": bits, "best": rec, "elite": np.array(hist_e, dtype=np.int32),
           "elite_fitness": np.array(hist_f, dtype=np.int64), "fitness": fit}
    if n * ng <= 1 << 14:
        out["state"] = k.to(torch.int16).cpu().numpy()
    return out
