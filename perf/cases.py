"""What a program asks of this library, as cases that can be timed and compared.

Every case calls the public entry points as a user's program does, on inputs
made from a seed.  Instances follow the synthetic workload family of this
repository (integer coordinates on [0, 1000]^2, uniform or clustered; fleets of
about one vehicle per 25-50 customers; the processing-time variants base, 2x,
5x, 1R10 and 1R20).  Results are whole numbers (makespans, status bits, routes,
counts) or copies of keys, the same on every run of the same inputs.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

import paper_2602_23685_gb300 as vrp


def listed():
    return [
        # one neighbourhood or one small population scored in a loop: the call itself is the cost
        dict(name="eval_n16_call", kind="eval", n=16, m=2, R=4, Q=4, p="base", clustered=False, full=False,
             num=256, bits=32, cyclic=0.0, tune=False),
        # a population of mid-size candidates, all feasible orders (decoder or ALNS output)
        dict(name="eval_n100_m4", kind="eval", n=100, m=4, R=10, Q=5, p="2x", clustered=False, full=False,
             num=65536, bits=32, cyclic=0.0, tune=False),
        # odd sizes, vehicles leaving full, a quarter of the candidates in random order (most of those
        # deadlock): what unrepaired perturbation produces
        dict(name="eval_n499_mixed", kind="eval", n=499, m=19, R=152, Q=8, p="1R10", clustered=True, full=True,
             num=65536, bits=32, cyclic=0.25, tune=False),
        # the full-size batch of a program that scores millions and tunes the shape once
        dict(name="eval_n1000_tuned", kind="eval", n=1000, m=20, R=100, Q=10, p="1R20", clustered=False, full=False,
             num=262144, bits=32, cyclic=0.0, tune=True),
        # candidates produced on the host: pinned 16-bit buffers in, makespans out
        dict(name="eval16_host_n1000", kind="host", n=1000, m=20, R=100, Q=10, p="1R20", clustered=True, full=False,
             num=32768, bits=16, cyclic=0.0, tune=False),
        # many customers' instances of uneven size in one launch
        dict(name="multi_32", kind="multi", instances=32, n_lo=17, n_hi=500, Q=8, p="1R10", num=4096),
        # coordination metrics of a population of complete solutions
        dict(name="coordination_n200", kind="coord", n=200, m=6, R=20, Q=6, p="5x", clustered=True, num=32768),
        # decoding a population of the paper's 4n chromosomes
        dict(name="decode_n200_hints", kind="decode", n=200, m=6, R=20, Q=6, p="5x", clustered=True, num=1024,
             layout=1),
        # warm-started BRKGA
        dict(name="brkga_n200", kind="brkga", n=200, m=6, R=20, Q=6, p="5x", clustered=True, pop=1024, gens=30,
             layout=0),
        # ALNS on one large instance, from the library's own start
        dict(name="alns_n1000", kind="alns", n=1000, m=20, R=100, Q=10, p="1R20", clustered=False, iters=20,
             replicas=1, destroy=1, repair=3, refine=0),
        # multi-instance ALNS with every operator, the local search and checkpoints
        dict(name="alns_n120_x8", kind="alns", n=120, m=5, R=12, Q=5, p="2x", clustered=True, iters=60,
             replicas=8, destroy=63, repair=15, refine=2),
        # a burst of solve requests, each ALNS then BRKGA, on four concurrent slots
        dict(name="serve_8", kind="serve", requests=8, n_lo=50, n_hi=300, Q=10, p="1R20", iters=40, pop=256, gens=20),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "eval", "host", "multi", "coord", "decode", "brkga", "alns", "alns",
                       "serve"])
    p = rng.choice(["base", "2x", "5x", "1R10", "1R20"])
    if kind == "multi":
        return dict(kind=kind, instances=rng.randint(8, 32), n_lo=17, n_hi=_log_int(rng, 60, 500), Q=8, p=p,
                    num=_log_int(rng, 512, 4096))
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(4, 8), n_lo=50, n_hi=rng.randint(80, 300), Q=10, p=p,
                    iters=rng.randint(10, 40), pop=256, gens=rng.randint(5, 20))
    n = _log_int(rng, 16, 1000)
    m = max(1, min(24, -(-n // rng.randint(20, 50)) + rng.randint(0, 2)))
    R, Q = max(m, -(-n // 10)), rng.randint(4, 10)
    c = dict(kind=kind, n=n, m=m, R=R, Q=Q, p=p, clustered=rng.random() < 0.5)
    if kind in ("eval", "host"):
        full = rng.random() < 0.25
        most = max(1024, min(262144, (250 << 20 if kind == "host" else 1 << 30) // (8 * n)))
        c.update(full=full, R=m * Q if full else R, num=_log_int(rng, 256, most), bits=rng.choice([16, 32]),
                 cyclic=rng.choice([0.0, 0.0, 0.1, 0.25]), tune=False)
    elif kind == "coord":
        c.update(num=_log_int(rng, 512, max(2048, min(32768, (64 << 20) // (8 * n)))))
    elif kind == "decode":
        c.update(n=min(n, 500), num=_log_int(rng, 128, 1024), layout=rng.randint(0, 1))
    elif kind == "brkga":
        c.update(n=min(n, 250), pop=_log_int(rng, 256, 1024), gens=rng.randint(5, 30), layout=rng.randint(0, 1))
    else:
        replicas = rng.choice([1, 1, 4, 8]) if n <= 200 else 1
        c.update(iters=rng.randint(5, 20), replicas=replicas, destroy=rng.choice([1, 15, 63]),
                 repair=rng.choice([1, 3, 7]), refine=0)
    return c


# ---- inputs -----------------------------------------------------------------
def _instance(n, m, R, Q, p, clustered, seed):
    g = np.random.default_rng([seed & 0x7fffffff, n, m])
    if clustered:
        centres = g.integers(0, 1001, size=(8, 2)).astype(np.float64)
        xy = centres[g.integers(0, 8, size=n + 1)] + g.normal(0.0, 60.0, size=(n + 1, 2))
        coords = np.clip(np.rint(xy), 0, 1000).astype(np.int32)
    else:
        coords = g.integers(0, 1001, size=(n + 1, 2)).astype(np.int32)
    if p in ("base", "2x", "5x"):
        times = g.integers(50, 151, size=n) * {"base": 1, "2x": 2, "5x": 5}[p]
    else:
        mean = float(np.mean(np.hypot(*(coords[1:] - coords[0]).astype(np.float64).T)))
        times = np.rint(g.integers(1, 11, size=n) * mean / 5.0) if p == "1R10" else \
            np.rint(g.integers(1, 21, size=n) * mean / 10.0)
    return types.SimpleNamespace(n=n, m=m, R=R, Q=Q, coords=np.ascontiguousarray(coords, dtype=np.int32),
                                 p=np.ascontiguousarray(times, dtype=np.int32))


def _candidates(n, m, num, cyclic, seed, dtype):
    """num x 2n op codes and num x (m+1) offsets on the GPU: a random order of
    all ops with every drop before its pickup (the last `cyclic` share in plain
    random order), each op on a random vehicle, routes in that order."""
    g = torch.Generator(device="cuda").manual_seed(seed & 0x7fffffff)
    ops = torch.empty((num, 2 * n), dtype=dtype, device="cuda")
    off = torch.zeros((num, m + 1), dtype=dtype, device="cuda")
    rows = max(1, (32 << 20) // (2 * n))
    ordered = num - int(num * cyclic)
    for a in range(0, num, rows):
        b = min(num, a + rows)
        at = torch.randint(0, 1 << 25, (b - a, n, 2), generator=g, device="cuda", dtype=torch.int32)
        k = max(0, min(b, ordered) - a)
        at[:k] = at[:k].sort(dim=2).values
        veh = torch.randint(0, m, (b - a, 2 * n), generator=g, device="cuda", dtype=torch.int32)
        key = (veh << 25) | at.view(b - a, 2 * n)
        ops[a:b] = (key.sort(dim=1, stable=True).indices + 2).to(dtype)
        count = torch.zeros((b - a, m), dtype=torch.int32, device="cuda")
        count.scatter_add_(1, veh.long(), torch.ones_like(veh))
        off[a:b, 1:] = count.cumsum(1).to(dtype)
    return ops, off


def _make(case, w):
    return vrp.Instance.from_workload(w, load_full=case.get("full", False))


def _sizes(case):
    """n spread over [n_lo, n_hi] by its logarithm, small and large ones in turn."""
    count = case.get("instances") or case["requests"]
    lo, hi = case["n_lo"], case["n_hi"]
    sizes = [int(round(lo * (hi / lo) ** (i / (count - 1)))) for i in range(count)]
    return sizes[0::2] + sizes[1::2]


def _requests(case, seed):
    """Instances of uneven size, one vehicle per 25 customers, a pool of a tenth of them."""
    return [_instance(n, -(-n // 25), -(-n // 10), case["Q"], case["p"], "requests" in case and i % 2 == 1, seed + i)
            for i, n in enumerate(_sizes(case))]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case, seed=int(seed))
    if kind == "multi":
        items = []
        for i, w in enumerate(_requests(case, seed)):
            ops, off = _candidates(w.n, w.m, case["num"], 0.0, seed + 1000 + i, torch.int32)
            items.append((vrp.Instance.from_workload(w), ops, off))
        s["plan"] = vrp.MultiBatch(items)
        return s
    if kind == "serve":
        s["work"] = _requests(case, seed)
        s["server"] = vrp.Server(8 << 30, max_active=4)
        return s
    w = _instance(case["n"], case["m"], case["R"], case["Q"], case["p"], case["clustered"], seed)
    s["inst"] = _make(case, w)
    if kind in ("eval", "host", "coord"):
        dtype = torch.int16 if case.get("bits") == 16 else torch.int32
        s["ops"], s["off"] = _candidates(case["n"], case["m"], case["num"], case.get("cyclic", 0.0), seed, dtype)
        if kind == "host":
            s["ops"], s["off"] = s["ops"].cpu().pin_memory(), s["off"].cpu().pin_memory()
            s["z"] = torch.empty(case["num"], dtype=torch.int32).pin_memory()
            s["st"] = torch.empty(case["num"], dtype=torch.int32).pin_memory()
        elif kind == "eval" and case["tune"]:
            head = min(case["num"], 32768)
            vrp.autotune(s["inst"], s["ops"][:head], s["off"][:head])
    elif kind == "decode":
        g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7fffffff)
        s["keys"] = torch.rand((case["num"], vrp.key_length(s["inst"], case["layout"])), generator=g, device="cuda")
    elif kind == "brkga":
        ops, off, _ = vrp.initial_solution_paper(s["inst"], 0)
        s["warm"] = (ops, off)
        s["params"] = vrp.brkga_params(case["pop"], case["gens"], layout=case["layout"])
    elif kind == "alns":
        s["params"] = vrp.alns_params(case["iters"], repair_mask=case["repair"], destroy_mask=case["destroy"],
                                      replicas=case["replicas"], sync_every=20, ls_pickup_every=20,
                                      ls_relocate_every=50, init_refine_rounds=case["refine"])
    return s


# ---- one pass -----------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "eval":
        return vrp.evaluate(s["inst"], s["ops"], s["off"])
    if kind == "host":
        return vrp.evaluate_host(s["inst"], s["ops"], s["off"], s["z"], s["st"])
    if kind == "multi":
        return s["plan"].evaluate()
    if kind == "coord":
        return vrp.coordination(s["inst"], s["ops"], s["off"])
    if kind == "decode":
        return vrp.brkga_decode(s["inst"], s["keys"], layout=s["layout"])
    if kind == "brkga":
        r = vrp.brkga_run(s["inst"], s["params"], seed=s["seed"], warm=s["warm"], final_keys=True)
        return [r["best_ops"], r["best_off"], r["z_best"], r["best_fitness"], r["trace"], r["keys"]]
    if kind == "alns":
        r = vrp.alns_run(s["inst"], s["params"], seed=s["seed"])
        st = r["stats"]
        counts = [st.accepted, st.improved, st.new_best, st.reheats, st.rejected_infeasible, st.ls_moves, st.imports]
        return [r["best_ops"], r["best_off"], r["z_best"], r["cur_ops"], r["cur_off"], r["z_current"], r["traces"],
                counts]
    ids = [s["server"].submit(w, alns_iterations=s["iters"], brkga_pop=s["pop"], brkga_generations=s["gens"],
                              seed=s["seed"] + i, init_refine_rounds=0) for i, w in enumerate(s["work"])]
    out = []
    for k in ids:
        r = s["server"].wait(k)
        out.append([r["ops"], r["off"], np.array([r["status"], r["z_alns"], r["z_brkga"], r["z_best"]])])
    return out


def exact(case, seed):
    # whole numbers throughout (the returned keys are drawn 24-bit fractions, copied and never computed with)
    return None


# ---- what a pass cannot do without ---------------------------------------------
def _eval_work(n, m, num, size):
    # codes and offsets in, two words out; per op a leg (two differences, two
    # products, the root), the arrival, the wait and the stock
    return num * (size * (2 * n + m + 1) + 8) + 12 * (n + 1), num * 2 * n * 8


def _decode_work(n, m, num, length):
    # the sort's comparisons, and per op the arrival and the choice over all vehicles
    return num * (4 * length + 4 * (2 * n + m + 1) + 16), num * 2 * n * (math.log2(2 * n) + 2 * m)


def _alns_work(n, m, iters):
    # per inserted customer: the longest-path table's update and every gap's row
    # and column terms for the customers still out
    q = max(4, int(0.05 * n)) * 0.75
    N = 2 * n
    return 8 * N + 12 * n, iters * q * (2 * N * N + (q / 2) * 2 * (N + m) * 6)


def work(case):
    kind = case["kind"]
    if kind in ("multi", "serve"):
        b = f = 0
        for n in _sizes(case):
            m = -(-n // 25)
            if kind == "multi":
                bi, fi = _eval_work(n, m, case["num"], 4)
            else:
                b1, f1 = _alns_work(n, m, case["iters"])
                b2, f2 = _decode_work(n, m, case["pop"] * case["gens"], 2 * n + m)
                bi, fi = b1 + b2, f1 + f2
            b, f = b + bi, f + fi
        return {"bytes": b, "flops": f}
    n, m = case["n"], case["m"]
    if kind in ("eval", "host"):
        b, f = _eval_work(n, m, case["num"], case["bits"] // 8)
    elif kind == "coord":
        b, f = _eval_work(n, m, case["num"], 4)
    elif kind == "decode":
        b, f = _decode_work(n, m, case["num"], 4 * n if case["layout"] else 2 * n + m)
    elif kind == "brkga":
        b, f = _decode_work(n, m, case["pop"] * case["gens"], 4 * n if case["layout"] else 2 * n + m)
    else:
        b, f = _alns_work(n, m, case["iters"] * case["replicas"])
    return {"bytes": b, "flops": f}
