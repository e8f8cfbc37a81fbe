"""What this framework is measured on: the calls its users make, over the range of sizes they make them with.

Four kinds of call, each through the binding's public entry points:

  run        a whole run of the method on loaded shards: x^0, the initial g_i (Algorithm 2, input line), T iterations in
             one call, the state read back.  Shards from a few hundred rows to more than the L2 holds, rows from 16 to
             some thousands of columns, both objectives, Algorithms 2, 3 (EF21+) and 4 (EF).
  minibatch  the same with sampled rows (Algorithm 5), the lists of all iterations drawn beforehand.
  round      rounds on gradients that the caller supplies (a training loop that brings its own model): n vectors of
             some thousands to some millions of entries, Algorithms 2, 3, 4 and the scaled Rand-k compressor, then a
             checkpoint of the state.
  topk       the compressor alone on a batch of vectors.
"""
import math

import torch

from paper_2106_05203_b200 import binding as B

LAM = 0.1                          # the regulariser weight of the logistic workloads
L2_BYTES = 126 << 20               # shards beyond this come from HBM in every iteration
VARIANTS = {"ef21": B.VARIANT_EF21, "plus": B.VARIANT_EF21_PLUS, "ef": B.VARIANT_EF}


def listed():
    return [
        # the smallest workload of the repository (4 workers, 200 dense rows, Top-4, its own 100 iterations): latency
        {"name": "run_tiny", "op": "run", "method": "ef21", "objective": "logistic", "features": "gauss", "density": 1.0,
         "sorted": False, "n": 4, "d": 64, "rows": 200, "k": 4, "steps": 100},
        # the headline workload: mushrooms-shaped, 20 workers, Top-1, shards that stay on chip
        {"name": "run_mushrooms", "op": "run", "method": "ef21", "objective": "logistic", "features": "bernoulli", "density": 0.19,
         "sorted": False, "n": 20, "d": 112, "rows": 8124, "k": 1, "steps": 100},
        # a9a-shaped with larger messages
        {"name": "run_a9a_top16", "op": "run", "method": "ef21", "objective": "logistic", "features": "bernoulli", "density": 0.11,
         "sorted": False, "n": 20, "d": 123, "rows": 32561, "k": 16, "steps": 50},
        # w8a-shaped, heterogeneous split (rows sorted by label), 60 MB of shards
        {"name": "run_w8a", "op": "run", "method": "ef21", "objective": "logistic", "features": "bernoulli", "density": 0.04,
         "sorted": True, "n": 20, "d": 300, "rows": 49749, "k": 1, "steps": 50},
        # the same rows, ten times as many: 600 MB, read from HBM in every iteration
        {"name": "run_beyond_l2", "op": "run", "method": "ef21", "objective": "logistic", "features": "bernoulli", "density": 0.04,
         "sorted": False, "n": 20, "d": 300, "rows": 500000, "k": 1, "steps": 20},
        # least squares on wide dense rows (an odd number of columns), 1 % of the entries per message
        {"name": "run_wide", "op": "run", "method": "ef21", "objective": "least_squares", "features": "gauss", "density": 1.0,
         "sorted": False, "n": 20, "d": 5001, "rows": 6000, "k": 50, "steps": 20},
        # stochastic iterations, 32 rows per worker
        {"name": "minibatch_mushrooms", "op": "minibatch", "features": "bernoulli", "density": 0.19,
         "n": 20, "d": 112, "rows": 8124, "k": 1, "tau": 32, "steps": 100},
        # the compressor alone: one short vector, a batch of medium ones, one of the size of a model
        {"name": "topk_short", "op": "topk", "values": "gauss", "batch": 1, "d": 1000, "k": 10},
        {"name": "topk_medium", "op": "topk", "values": "student", "batch": 20, "d": 70001, "k": 700},
        {"name": "topk_model", "op": "topk", "values": "student", "batch": 1, "d": 25000001, "k": 25000},
        # the compressor and aggregation stress workload: 64 workers, 4 million entries each, k = d / 1000
        {"name": "round_stress", "op": "round", "method": "ef21", "n": 64, "d": 4194304, "k": 4194, "steps": 10},
        # EF21+ on supplied gradients: 16 workers, a million entries (odd), 1 % of them per message
        {"name": "round_plus", "op": "round", "method": "plus", "n": 16, "d": 1000003, "k": 10000, "steps": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case; how often each kind comes up follows the listed ones.  Bounded so that it costs no more than the
    largest of them (entries read over the whole call)."""
    while True:
        kind = rng.choice(["run_small"] * 4 + ["run_large"] * 2 + ["minibatch"] + ["topk"] * 3 + ["round"] * 2)
        if kind == "run_small":
            # shards that stay on chip or in L2, rows of at most 512 columns
            n, d = rng.choice([2, 5, 10, 20, 20, 31, 50, 100]), _log_int(rng, 16, 512)
            rows = n * _log_int(rng, 30, 2500) + rng.randrange(n)
            features = rng.choice(["bernoulli", "bernoulli", "gauss"])
            case = {"op": "run", "method": rng.choice(["ef21", "ef21", "ef21", "plus", "ef"]),
                    "objective": rng.choice(["logistic", "logistic", "logistic", "least_squares"]), "features": features,
                    "density": round(rng.uniform(0.04, 0.2), 3) if features == "bernoulli" else 1.0, "sorted": rng.random() < 0.25,
                    "n": n, "d": d, "rows": rows, "k": min(d // 4, rng.choice([1, 1, 1, 2, 4, 8, 16])), "steps": _log_int(rng, 10, 60)}
            if rows * d > 16000000:
                continue
        elif kind == "run_large":
            # wide rows, or more rows than the L2 holds
            if rng.random() < 0.5:
                n, d = rng.choice([4, 10, 20, 50]), _log_int(rng, 513, 8000)
                rows = n * _log_int(rng, 50, 1000) + rng.randrange(n)
                k = max(1, int(d * rng.choice([0.001, 0.01, 0.05])))
            else:
                n, d = rng.choice([10, 20, 37]), _log_int(rng, 64, 512)
                rows = n * _log_int(rng, 3000, 40000) + rng.randrange(n)
                k = rng.choice([1, 1, 4, 16])
            features = rng.choice(["bernoulli", "gauss"])
            case = {"op": "run", "method": rng.choice(["ef21", "ef21", "ef21", "plus", "ef"]),
                    "objective": rng.choice(["logistic", "least_squares"]), "features": features,
                    "density": round(rng.uniform(0.04, 0.2), 3) if features == "bernoulli" else 1.0, "sorted": rng.random() < 0.25,
                    "n": n, "d": d, "rows": rows, "k": k, "steps": rng.randint(5, 20)}
            if rows * d * case["steps"] > 2000000000:
                continue
        elif kind == "minibatch":
            n, d, tau = rng.choice([5, 10, 20, 40]), _log_int(rng, 16, 700), _log_int(rng, 8, 256)
            features = rng.choice(["bernoulli", "gauss"])
            case = {"op": "minibatch", "features": features,
                    "density": round(rng.uniform(0.04, 0.2), 3) if features == "bernoulli" else 1.0, "n": n, "d": d,
                    "rows": n * _log_int(rng, 300, 2500) + rng.randrange(n), "k": rng.choice([1, 1, 4]), "tau": tau,
                    "steps": _log_int(rng, 10, 100)}
        elif kind == "topk":
            batch, d = rng.choice([1, 1, 1, 4, 20, 64]), _log_int(rng, 100, 30000000)
            if batch * d > 60000000:
                continue
            case = {"op": "topk", "values": rng.choice(["gauss", "student"]), "batch": batch, "d": d,
                    "k": max(1, int(d * rng.choice([0.001, 0.01, 0.1])))}
        else:
            n, d = rng.choice([4, 8, 16, 20, 64]), _log_int(rng, 5000, 4500000)
            case = {"op": "round", "method": rng.choice(["ef21", "ef21", "plus", "ef", "randk"]), "n": n, "d": d,
                    "k": max(1, int(d * rng.choice([0.001, 0.01]))), "steps": rng.randint(1, 10)}
            if n * d > 268435456 or n * d * case["steps"] > 600000000 or (case["method"] == "plus" and d * case["steps"] > 5000000):
                continue
        return case


def _vectors(gen, count, d, values):
    """[count, d] supplied gradients: normal, or Student-t with three degrees of freedom; each with a scale in U(0.5, 2)."""
    out = torch.empty((count, d), dtype=torch.float32, device="cuda")
    for i in range(count):
        out[i].normal_(generator=gen)
        if values == "student":
            chi2 = torch.zeros(d, dtype=torch.float32, device="cuda")
            for _ in range(3):
                chi2 += torch.empty_like(chi2).normal_(generator=gen).square_()
            out[i] *= (3.0 / chi2).sqrt_()
        out[i] *= torch.empty(1, device="cuda").uniform_(0.5, 2.0, generator=gen)
    return out


def _shards(case, gen):
    """Rows, labels of a planted model (5 % flipped), shard boundaries and a stepsize 1/L from the features' distribution."""
    N, d, n = case["rows"], case["d"], case["n"]
    A = torch.empty((N, d), dtype=torch.float32, device="cuda")
    if case["features"] == "gauss":
        A.normal_(generator=gen)
        top = (1.0 + math.sqrt(d * n / N)) ** 2                      # largest eigenvalue of A_i^T A_i / m_i
    else:
        p = case["density"]
        A.bernoulli_(p, generator=gen)
        top = p * p * d + p * (1.0 - p) * (1.0 + math.sqrt(d * n / N)) ** 2
    w = torch.empty(d, device="cuda").normal_(generator=gen)
    y = torch.where((A * w).sum(1) >= 0, 1.0, -1.0)
    y = torch.where(torch.empty(N, device="cuda").uniform_(generator=gen) < 0.05, -y, y)
    if case.get("sorted"):
        order = torch.argsort(y, stable=True)
        A, y = A[order].contiguous(), y[order].contiguous()
    offsets = [i * (N // n) for i in range(n)] + [N]
    logistic = case.get("objective", "logistic") == "logistic"
    lam = LAM if logistic else 0.0
    gamma = 1.0 / ((0.25 if logistic else 2.0) * top + 2.0 * lam)
    return A, y, offsets, gamma, lam


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["op"] == "topk":
        return {"case": case, "v": _vectors(gen, case["batch"], case["d"], case["values"])}
    n, d, k = case["n"], case["d"], case["k"]
    s = {"case": case, "x0": torch.zeros(d, dtype=torch.float32, device="cuda")}
    if case["op"] == "round":
        s["V"] = _vectors(gen, n, d, "student")
        h = B.EF21(n, d, k, 0.01)
        if case["method"] == "randk":
            # per step and worker, one coordinate out of each of k equal strata: distinct and ascending
            width = d // k
            pick = torch.randint(0, width, (case["steps"], n, k), generator=gen, device="cuda")
            s["sets"] = (pick + width * torch.arange(k, device="cuda")).to(torch.int32).contiguous()
        else:
            h.set_variant(VARIANTS[case["method"]])
    else:
        A, y, offsets, gamma, lam = _shards(case, gen)
        h = B.EF21(n, d, k, gamma, lam, total_rows=case["rows"])
        if case["op"] == "run":
            h.set_variant(VARIANTS[case["method"]])
            h.set_objective(B.OBJECTIVE_LOGISTIC if case["objective"] == "logistic" else B.OBJECTIVE_LEAST_SQUARES)
        else:
            s["batches"] = torch.randint(0, case["rows"] // n, (case["steps"], n, case["tau"]), generator=gen, device="cuda",
                                         dtype=torch.int32)
        h.load_shards(A, y, offsets)
    s["h"] = h
    return s


def run(state):
    case = state["case"]
    if case["op"] == "topk":
        return B.topk(state["v"], case["k"])
    h = state["h"]
    h.set_x(state["x0"])
    if case["op"] == "round":
        h.init_grads(None, B.INIT_ZERO)
        if case["method"] == "randk":
            h.step_randk(state["sets"], state["V"])
        else:
            h.step_grads(state["V"], case["steps"])
        return h.get_state(messages=True)
    # Algorithm 4 starts from zero errors, the others from the compressed local gradients
    h.init(B.INIT_ZERO if case.get("method") == "ef" else B.INIT_COMPRESSED)
    if case["op"] == "minibatch":
        h.step_minibatches(state["batches"])
    else:
        h.step(case["steps"])
    # g is the mean of the g_i: near a stationary point only their rounding is left of it, so x and the g_i are compared
    x, _, gi, _, _ = h.get_state(messages=False)
    return x, gi


def work(case):
    if case["op"] == "topk":
        size = case["batch"] * case["d"]
        return {"bytes": 4 * size + 8 * case["batch"] * case["k"], "flops": size}
    n, d, k, steps = case["n"], case["d"], case["k"], case["steps"]
    state = 4 * (n * d + 2 * d)                                       # g_i, g and x, written once
    if case["op"] == "round":
        # every round needs V and g_i whole (with Rand-k only the drawn entries), x and g read and written
        per_round = 20 * n * k if case["method"] == "randk" else 8 * n * d
        return {"bytes": steps * (per_round + 16 * d) + 2 * state, "flops": steps * 3 * n * d}
    if case["op"] == "minibatch":
        rows = min(case["rows"], steps * n * case["tau"])
        return {"bytes": 4 * (rows + case["rows"]) * (d + 1) + 4 * steps * n * case["tau"] + state,
                "flops": 4 * (steps * n * case["tau"] + case["rows"]) * d}
    shards = 4 * case["rows"] * (d + 1)
    passes = steps + (0 if case["method"] == "ef" else 1)             # one more for the initial gradients
    return {"bytes": shards * (passes if shards > L2_BYTES else 1) + state, "flops": 4 * passes * case["rows"] * d}


def tolerance(case):
    # Selection and state updates are exact given the gradients; the local gradients are 32-bit sums whose order is free,
    # and an iteration builds on the one before.  (Iterations per call are kept to where Top-k picks do not hang on the
    # last bits of a gradient: after some hundreds two correct implementations part.)
    return "exact" if case["op"] in ("topk", "round") else {"rel": 1e-4}
