"""Performance cases of the routing simulator: the calls that its users make, over the range of sizes they make them at.

Four kinds, one for each part of the path, all through the package's public calls:

* ``score``   -- ``ctr.ctr_score_batch``: the standalone scorer, from one admission tick of a proxy to millions of requests.
* ``trace``   -- ``ctr.ctr_gen_trace``: synthetic traces, from the one replica of a saturation probe to a whole sweep.
* ``sim``     -- ``sweep.run_step``: simulation with checksum and goodput, with the trace made in the same step
  (``gen``) or in hand, as when one trace serves several simulations.
* ``goodput`` -- ``ctr.ctr_goodput`` with the P99 TPOT: Table 2's columns of a finished simulation.

Loads stay below the pools' saturation (or the structures are deep enough for the overload), so that every simulated
row completes: the outputs of a row that overflows are unspecified.
"""
import math

import torch

from paper_2609_16206_gb300 import ctr, sweep
from paper_2609_16206_gb300 import workloads as W

DEV = "cuda"
# requests per second that one prefill / one decode instance of the default cluster sustains, per trace law
# (mean prefill 20 ms + 0.15 ms x E[p]; decode at the batch that fills the KV capacity)
PREFILL_RPS = {"mixed": 6.8, "chat": 6.8, "reasoning": 6.8, "document": 2.8, "scarce": 6.8}
DECODE_RPS = {"mixed": 6.0, "chat": 18.0, "reasoning": 2.2, "document": 14.0, "scarce": 4.0}
POLICIES = {"four": W.ALL_POLICIES, "learned": (W.POLICY_LEARNED,), "baselines": W.ALL_POLICIES[1:],
            "five": W.ALL_POLICIES + (W.POLICY_LEARNED_P2,)}


def listed():
    return [
        # a proxy's admission tick: a few hundred queued requests against an eight-instance pool
        {"name": "score_tick", "kind": "score", "n": 257, "inst": 8, "shift": 0},
        # the scorer's standing workload: 2^20 requests x 64 instances
        {"name": "score_batch", "kind": "score", "n": 1 << 20, "inst": 64, "shift": 0},
        # an offline what-if over a large fleet: a ragged request count, a wide pool, tens of MB in and out
        {"name": "score_fleet", "kind": "score", "n": 6_000_003, "inst": 200, "shift": 0},
        # one probe of a saturation search: a single Poisson replica
        {"name": "trace_probe", "kind": "trace", "replicas": 1, "n": 10_000, "mmpp": False, "classes": 2},
        # the trace of a whole sweep: bursty arrivals, three seeds
        {"name": "trace_sweep", "kind": "trace", "replicas": 4096, "n": 20_000, "mmpp": True, "classes": 2},
        # the single-replica comparison of the four policies on a small pool, its trace in hand
        {"name": "sim_single", "kind": "sim", "law": "mixed", "pre": 1, "dec": 3, "replicas": 1, "n": 2000, "load": 0.6,
         "mmpp": False, "policies": "four", "sets": 1, "deployed": False, "gen": False},
        # the deployed proxy's signals (ledger backlog, 50 ms poll), every policy, bursty arrivals
        {"name": "sim_deployed", "kind": "sim", "law": "mixed", "pre": 2, "dec": 6, "replicas": 256, "n": 10_000,
         "load": 0.55, "mmpp": True, "policies": "five", "sets": 1, "deployed": True, "gen": True},
        # the document family: batched prefill, long prompts, short outputs
        {"name": "sim_document", "kind": "sim", "law": "document", "pre": 2, "dec": 6, "replicas": 250, "n": 10_000,
         "load": 0.9, "mmpp": False, "policies": "four", "sets": 1, "deployed": False, "gen": True},
        # one pool width of the calibration study: the learned router under 65 constant sets on the same traces
        {"name": "sim_calibration", "kind": "sim", "law": "mixed", "pre": 2, "dec": 5, "replicas": 48, "n": 10_000,
         "load": 0.8, "mmpp": False, "policies": "learned", "sets": 65, "deployed": False, "gen": False},
        # the large pool under scarcity: 32 instances, three classes, 1.2 x what the prefill pool sustains
        {"name": "sim_large_pool", "kind": "sim", "law": "scarce", "pre": 4, "dec": 28, "replicas": 4096, "n": 5000,
         "load": 1.2, "mmpp": False, "policies": "four", "sets": 1, "deployed": False, "gen": True},
        # the replica sweep at full size: trace, four policies, checksum and goodput in one step
        {"name": "sim_sweep", "kind": "sim", "law": "mixed", "pre": 2, "dec": 6, "replicas": 4096, "n": 20_000,
         "load": 0.55, "mmpp": True, "policies": "four", "sets": 1, "deployed": False, "gen": True},
        # Table 2's columns over a quarter of that sweep: met count, P99 TTFT and P99 TPOT per row
        {"name": "goodput_table", "kind": "goodput", "replicas": 1024, "rows": 4, "n": 20_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("score", "trace", "sim", "sim", "sim", "goodput"))
    if kind == "score":
        # shift 1: the request arrays are a view that starts one element into a buffer
        return {"kind": kind, "n": _log(rng, 1, 6_000_000), "inst": _log(rng, 1, 256), "shift": rng.choice((0, 0, 0, 1))}
    if kind == "trace":
        n = _log(rng, 33, 20_000)
        return {"kind": kind, "replicas": _log(rng, 1, min(16_384, 80_000_000 // n)), "n": n,
                "mmpp": rng.random() < 0.5, "classes": rng.choice((1, 2, 3, 4))}
    if kind == "goodput":
        n = _log(rng, 50, 120_000)
        rows = rng.choice((1, 2, 3, 4, 5))
        return {"kind": kind, "replicas": _log(rng, 1, max(1, min(8192, 80_000_000 // (n * rows)))), "rows": rows, "n": n}
    law = rng.choice(("mixed", "mixed", "chat", "reasoning", "document", "scarce"))
    pre = rng.randint(1, 4)
    dec = rng.randint(3, 28) if law == "scarce" else rng.randint(1, 12)
    sets = rng.choice((1, 1, 1, 5, 65))
    policies = "learned" if sets > 1 else rng.choice(("four", "five", "learned", "baselines"))
    n = _log(rng, 500, 12_000)
    budget = 24_000_000 if pre + dec > 8 else 60_000_000
    most = max(1, budget // (n * sets * len(POLICIES[policies])))
    return {"kind": kind, "law": law, "pre": pre, "dec": dec, "replicas": _log(rng, 1, min(4096, most)), "n": n,
            "load": round(rng.uniform(0.3, 0.85), 3), "mmpp": rng.random() < 0.5, "policies": policies, "sets": sets,
            "deployed": rng.random() < 0.3, "gen": rng.random() < 0.5}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _trace_cfg(case, seed):
    """The trace law of a ``sim`` or ``trace`` case; 64 seeds apart, so that no replica is shared between seeds."""
    tc = {"chat": W.chat, "reasoning": W.reasoning, "document": W.document,
          "scarce": W.large_pool}.get(case.get("law"), W.replica_sweep)().trace
    if case["kind"] == "trace":
        rate, classes = 4.0, case["classes"]
        tc = tc.replace(n_classes=classes, class_thr=tuple(W.prob_to_u32_threshold((i + 1) / classes)
                                                           for i in range(classes - 1)))
    else:
        rate = case["load"] * min(case["pre"] * PREFILL_RPS[case["law"]], case["dec"] * DECODE_RPS[case["law"]])
    mreq = max(1, int(rate * 1000))
    rates = (max(1, int(0.4 * mreq)), int(1.6 * mreq) + 1) if case["mmpp"] else (mreq, mreq)
    return tc.replace(seed=int(seed) * 64, n_seeds=3 if case["mmpp"] else 1, arrival_kind=int(case["mmpp"]),
                      rate_mreq=rates, dwell_mean_us=10_000_000)


def _sim_cfg(case):
    if case["law"] == "scarce":
        return W.large_pool().sim.replace(n_prefill=case["pre"], n_decode=case["dec"])
    batch = W.PREFILL_BATCH_TOKENS if case["law"] == "document" else 0
    return W.SimCfg(n_prefill=case["pre"], n_decode=case["dec"], prefill_batch_tokens=batch)


def _const_sets(case):
    base = W.large_pool().consts[0] if case["law"] == "scarce" else W.CALIBRATED
    if case["deployed"]:
        base = W.as_deployed(base)
    return W.mispriced_sets(base)[:case["sets"]]


def _lengths(n, g):
    """Prompt and output lengths of the mixed law, as float64 whole numbers."""
    z = torch.randn((2, n), generator=g, device=DEV, dtype=torch.float64)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    p = torch.floor(torch.exp(W.LN_512 + z[0]) + 0.5).clamp_(16, 8192)
    o = torch.where(u < 0.7, W.LN_128 + 0.8 * z[1], W.LN_1024 + 0.6 * z[1])
    return p, torch.floor(torch.exp(o) + 0.5).clamp_(1, 4096)


def _prepare_score(case, seed):
    n, inst, sh, g = case["n"], case["inst"], case["shift"], _gen(seed)
    p, o = _lengths(n + sh, g)
    noise = torch.randn(n + sh, generator=g, device=DEV, dtype=torch.float64)
    oh = torch.floor(o * torch.exp(0.3 * noise) + 0.5).clamp_(1, 1 << 17)
    cls = (torch.rand(n + sh, generator=g, device=DEV) >= 0.6).to(torch.uint8)
    state = torch.rand((3, inst), generator=g, device=DEV)
    s = {"p": p.float()[sh:], "oh": oh.float()[sh:], "cls": cls[sh:],
         "Q": torch.floor(state[0] * 65537), "A": torch.floor(state[1] * 257), "kap": state[2].clone(),
         "argmin": torch.empty(n, dtype=torch.int32, device=DEV), "cost": torch.empty(n, dtype=torch.float32, device=DEV)}
    return s


def _prepare_goodput(case, seed):
    """A finished simulation's outputs, drawn: TTFTs around half a second, 15 to 60 ms per output token."""
    R, rows, n, g = case["replicas"], case["rows"], case["n"], _gen(seed)
    trace = ctr.empty_requests(R, n, DEV)
    t_first = torch.empty((R * rows, n), dtype=torch.int64, device=DEV)
    t_done = torch.empty_like(t_first)
    step = max(1, 8_000_000 // n)  # replicas at a time: bounds the temporaries
    for r0 in range(0, R, step):
        m = min(step, R - r0)
        p, o = _lengths(m * n, g)
        gaps = torch.empty((m, n), device=DEV, dtype=torch.float64).exponential_(1 / 133_000.0, generator=g)
        arrival = torch.cumsum(gaps.long(), 1)
        trace["arrival_us"][r0:r0 + m] = arrival
        trace["prompt_len"][r0:r0 + m] = p.view(m, n).int()
        trace["true_out"][r0:r0 + m] = o.view(m, n).int()
        trace["pred_out"][r0:r0 + m] = o.view(m, n).int()
        trace["slo_class"][r0:r0 + m] = (torch.rand((m, n), generator=g, device=DEV) >= 0.6).to(torch.uint8)
        for j in range(rows):
            row = slice(r0 * rows + j, (r0 + m) * rows, rows)
            ttft = torch.exp(13.1 + 0.8 * torch.randn((m, n), generator=g, device=DEV))
            tpot = 15_000 + 45_000 * torch.rand((m, n), generator=g, device=DEV)
            first = arrival + ttft.long()
            t_first[row] = first
            t_done[row] = first + (tpot.double() * (o.view(m, n) - 1)).long()
    out = {k: torch.empty(R * rows, dtype=torch.int64, device=DEV) for k in ("met", "p99_ttft", "p99_tpot")}
    return {"trace": trace, "t_first": t_first, "t_done": t_done, "sim": W.SimCfg(), "out": out}


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "score":
        s.update(_prepare_score(case, seed))
    elif case["kind"] == "goodput":
        s.update(_prepare_goodput(case, seed))
    elif case["kind"] == "trace":
        s["cfg"] = _trace_cfg(case, seed)
        s["trace"] = ctr.empty_requests(case["replicas"], case["n"], DEV)
    else:
        s["cfg"], s["sim"], s["sets"] = _trace_cfg(case, seed), _sim_cfg(case), _const_sets(case)
        s["policies"] = list(POLICIES[case["policies"]])
        n_rows = case["replicas"] * len(s["sets"]) * len(s["policies"])
        s["buf"] = sweep.alloc(s["sim"], case["replicas"], n_rows, case["n"], DEV)
        if not case["gen"]:
            ctr.ctr_gen_trace(s["cfg"], case["replicas"], 0, case["n"], s["buf"].trace)
    return s


# ---------------------------------------------------------------- the calls
def run(state):
    s, case = state, state["case"]
    if case["kind"] == "score":
        ctr.ctr_score_batch(s["p"], s["oh"], s["cls"], s["Q"], s["A"], s["kap"], W.SCORE_CONSTS, s["argmin"], s["cost"])
        return {"argmin": s["argmin"], "cost": s["cost"]}
    if case["kind"] == "trace":
        ctr.ctr_gen_trace(s["cfg"], case["replicas"], 0, case["n"], s["trace"])
        return s["trace"]
    if case["kind"] == "goodput":
        out = s["out"]
        ctr.ctr_goodput(s["sim"], s["trace"], case["replicas"], case["rows"], case["n"], s["t_first"], s["t_done"],
                        out["met"], out["p99_ttft"], p99_tpot_us=out["p99_tpot"])
        return out
    b = s["buf"]
    sweep.run_step(s["cfg"], s["sim"], s["sets"], s["policies"], case["replicas"], case["n"], 0, b, gen=case["gen"])
    return {"t_first": b.t_first, "t_done": b.t_done, "row_hash": b.row_hash, "row_status": b.row_status,
            "met": b.met, "p99_ttft": b.p99}


def work(case):
    if case["kind"] == "score":  # 9 B in and 8 B out a request; the instance state; one evaluation of the cost
        return {"bytes": 17 * case["n"] + 12 * case["inst"], "flops": 14 * case["n"]}
    if case["kind"] == "trace":  # 21 B a request
        return {"bytes": 21 * case["replicas"] * case["n"], "flops": 0}
    if case["kind"] == "goodput":  # arrival, output length and class once, both times of each row; three results a row
        return {"bytes": case["replicas"] * (13 * case["n"] + case["rows"] * (16 * case["n"] + 24)), "flops": 0}
    rows = case["sets"] * len(POLICIES[case["policies"]])
    return {"bytes": case["replicas"] * (21 * case["n"] + rows * (16 * case["n"] + 28)), "flops": 0}


def tolerance(case):
    """Everything but the scorer is whole numbers, defined to the last bit.  The scorer's cost is a dozen fp32 operations
    (against 64 bits over 42 inputs: 3e-8 to 7e-8 in the 2-norm, 2e-7 at most).  An argmin may differ where two
    instances' costs are within a few fp32 roundings of each other; predicted lengths are whole numbers, so all requests
    of one length (up to 0.3 % of them) stand at such a tie together (seen in none of the 42)."""
    if case["kind"] == "score":
        return {"rel": 3e-7, "max": 8e-7, "differ": min(0.01, max(4e-3, 2 / case["n"]))}
    return "exact"


# ---------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    if case["kind"] == "score":
        return _exact_score(case, seed)
    if case["kind"] == "goodput":
        return _exact_goodput(case, seed)
    return None  # defined as integer event order (sim) or as a fixed sequence of fp32 roundings (trace)


def _exact_score(case, seed):
    s = _prepare_score(case, seed)
    wb, ws, wq, rho, pre0, pre, dec, act, inv_c, *sigma = (float(x) for x in W.SCORE_CONSTS)
    Q, A, kap = (s[k].double() for k in ("Q", "A", "kap"))
    backlog, queue = wb * (pre * Q + act * A), wq * A
    sig = torch.tensor(sigma, dtype=torch.float64, device=DEV)
    argmin, cost = [], []
    for p, oh, c in zip(*(s[k].split(1 << 18) for k in ("p", "oh", "cls"))):
        p, oh, sg = p.double()[:, None], oh.double()[:, None], sig[c.long()][:, None]
        own = pre0 + pre * p + dec * oh * (1 + rho * (kap + (p + oh) * inv_c))
        best = (sg * (backlog + ws * own) + queue).min(1)
        argmin.append(best.indices.int())
        cost.append(best.values)
    return {"argmin": torch.cat(argmin), "cost": torch.cat(cost)}


def _exact_goodput(case, seed):
    s = _prepare_goodput(case, seed)
    n, rows, tr = case["n"], case["rows"], s["trace"]
    ttft_slo, tpot_slo = (torch.tensor(x, device=DEV) for x in (s["sim"].ttft_slo_us, s["sim"].tpot_slo_us))
    out = {"met": [], "p99_ttft": [], "p99_tpot": []}
    for r in range(case["replicas"]):
        first, done = (s[k][r * rows:(r + 1) * rows] for k in ("t_first", "t_done"))
        o, c = tr["true_out"][r].long(), tr["slo_class"][r].long()
        ttft, decode = first - tr["arrival_us"][r], done - first
        met = (ttft <= ttft_slo[c]) & ((o == 1) | (decode <= tpot_slo[c] * (o - 1)))
        out["met"].append(met.sum(1))
        out["p99_ttft"].append(ttft.sort(1).values[:, (99 * n + 99) // 100 - 1])
        many = o >= 2
        m = int(many.sum())
        if m == 0:
            out["p99_tpot"].append(torch.full((rows,), -1, device=DEV))
        else:
            tpot = decode[:, many] // (o[many] - 1)
            out["p99_tpot"].append(tpot.sort(1).values[:, (99 * m + 99) // 100 - 1])
    return {k: torch.cat(v) for k, v in out.items()}
