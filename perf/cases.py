"""What this simulator is used for, as cases that can be timed and compared.

A case is one sweep: `instances` request instances of up to `n` requests each,
simulated under a list of (policy, fairness budget) runs with `B` batch slots
and a KV cap of `kv` tokens.  `family` names the request distribution (those of
paper_2608_02244_gb300/workloads.py, drawn here on the GPU from the seed, with
the mean arrival gap `gap`; 0 = everything at step 0).  `epoch` picks the
event-driven kernel flag, `entry` the public call: the device-resident sweep
("async"), the numpy convenience call ("sweep"), the host-memory C entry point
("host") or the allocation-free one ("noalloc").  `per_request` asks for every
request's start and completion step too.
"""
from __future__ import annotations

import bisect
import heapq
import math

import numpy as np
import torch

from paper_2608_02244_gb300 import sim

INF = 2**31 - 1
C, TAU, P0 = 0.0005, 1e-6, 1.0 / 500.0

SWEEP = "fcfs:0,ljf:0,isjl:16,isjl:64,isjl:256,isjl:1024,isjl:%d" % INF
TINY = "isjl:0,isjl:1,isjl:2,isjl:4,isjl:%d" % INF
PROFIT = "fcfs:0,ljf:0," + ",".join("isjl:%d" % d for d in (50, 100, 150, 250, 300, 400, 500))

# per family: mean and largest planning length, and whether it is drawn with
# request counts (ragged) or upper-bound slack (robust)
FAMILIES = {
    "bimodal": (74, 288),      # short chat turns with a long minority
    "tiny": (7, 12),           # instances small enough for an exhaustive optimum
    "online": (1250, 6144),    # lognormal prompts and outputs
    "robust": (1400, 7168),    # the same with length predictions
    "heavy": (544, 9216),      # Pareto outputs
    "large": (2700, 49152),    # long-context lognormals
    "profit": (290, 1000),     # priced requests, some of which decline
}


def _case(name, family, instances, n, gap, B, kv, runs, epoch, entry, per_request):
    c = {"family": family, "instances": instances, "n": n, "gap": gap, "B": B, "kv": kv, "runs": runs,
         "epoch": epoch, "entry": entry, "per_request": per_request}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one short instance through the numpy call: a notebook or a unit test of a policy
        _case("single_200", "bimodal", 1, 200, 0.0, 32, 2048, "fcfs:0,ljf:0,isjl:32", False, "sweep", True),
        # one long trace: what a serving team replays, serial in time
        _case("trace_20000", "online", 1, 20000, 2.0, 256, 200000, "fcfs:0,isjl:256", False, "async", True),
        # thousands of tiny instances: checks against an exhaustive optimum
        _case("tiny_4096", "tiny", 4096, 6, 0.0, 3, 16, TINY, False, "async", True),
        # a few odd-sized instances inside another program's memory budget
        _case("noalloc_77x777", "online", 77, 777, 3.0, 48, 30011, "fcfs:0,sjf:0,isjl:200,isjl_beta:200", True,
              "noalloc", True),
        # all five policies side by side, odd sizes, a small batch
        _case("policies_1500x701", "heavy", 1500, 701, 1.0, 61, 40009,
              "fcfs:0,ljf:0,sjf:0,isjl:128,isjl_beta:128", False, "async", True),
        # instances too long for the in-memory sort, few of them
        _case("mid_96x9001", "large", 96, 9001, 0.4, 100, 400000, "fcfs:0,ljf:0,isjl:256", True, "async", True),
        # the profit experiment: ragged instances, nine runs, records only
        _case("profit_10000", "profit", 10000, 400, 0.0, 50, INF, PROFIT, False, "async", False),
        # the fairness-budget sweep, default kernel, with per-request steps
        _case("sweep_10000x1000", "online", 10000, 1000, 2.0, 256, 200000, SWEEP, False, "async", True),
        # the same sweep from host memory, event-driven kernel: records come back
        _case("sweep_host", "online", 10000, 1000, 2.0, 256, 200000, SWEEP, True, "host", False),
        # length predictions, event-driven kernel
        _case("robust_3000x1000", "robust", 3000, 1000, 2.0, 256, 200000, SWEEP, True, "async", True),
        # heavy-tailed offline mix, the most tasks of any workload
        _case("heavy_100000x500", "heavy", 100000, 500, 0.0, 128, 65536,
              "fcfs:0,ljf:0,isjl:32,isjl:128,isjl:512", True, "async", True),
        # a thousand long-context instances of 10^5 requests each
        _case("large_1024x100000", "large", 1024, 100000, 0.05, 512, 1000000, "fcfs:0,ljf:0,isjl:256", True,
              "async", True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more sweep of the listed ranges: instances from 6 to 10^5 requests,
    batches of 2 to 512, one instance to 10^5 of them, every policy and entry."""
    family = rng.choice(sorted(FAMILIES))
    mean, most = FAMILIES[family]
    n = 6 if family == "tiny" and rng.random() < 0.5 else _log(rng, 6, 100000)
    B = _log(rng, 2, 512) if n < 2000 else _log(rng, 64, 512)
    kv = rng.choice([INF, max(most, _log(rng, mean * max(2, B // 4), mean * B * 2))])
    # a run's steps stay in the listed range (time is serial within a run)
    conc = max(1.0, min(B, kv / mean))
    n = max(6, min(n, int(1.5e6 * conc / (2.5 * mean))))
    runs = []
    for _ in range(rng.randint(1, 7)):
        p = rng.choice(["fcfs", "ljf", "sjf", "isjl", "isjl", "isjl", "isjl_beta"])
        runs.append("%s:%d" % (p, rng.choice([INF, _log(rng, 1, max(2, most // 2))]) if "isjl" in p else 0))
    entry = rng.choice(["async", "async", "async", "sweep", "host", "noalloc"])
    total = {"sweep": 2e6, "noalloc": 1.5e6}.get(entry, 3e7)
    instances = _log(rng, 1, max(1, min(100000, total / n / (1 if entry != "async" else len(runs) / 3))))
    gap = rng.choice([0.0, round(math.exp(rng.uniform(math.log(0.05), math.log(8.0))), 3)])
    if family in ("profit", "bimodal", "tiny"):
        gap = 0.0
    return _case(None, family, instances, n, gap, B, kv, ",".join(runs), rng.random() < 0.5, entry,
                 entry in ("sweep", "noalloc") or (entry == "async" and rng.random() < 0.6))


# ------------------------------------------------------------------- inputs
def _lognormal(g, shape, median, sigma, lo, hi):
    x = torch.randn(shape, generator=g, device="cuda").mul_(sigma).add_(math.log(median)).exp_()
    return x.round_().clamp_(lo, hi).to(torch.int32)


def _uniform(g, shape, lo, hi):
    return torch.randint(lo, hi + 1, shape, generator=g, device="cuda", dtype=torch.int32)


def _inputs(case, seed):
    """(arrival, prompt, output, counts or None, slack or None), int32 on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    N, n, family = case["instances"], case["n"], case["family"]
    shape = (N, n)
    if case["gap"] > 0:
        gaps = torch.empty(shape, device="cuda", dtype=torch.float64).exponential_(1.0 / case["gap"], generator=g)
        arrival = gaps.cumsum_(1).floor_().to(torch.int32)
        del gaps
    else:
        arrival = torch.zeros(shape, device="cuda", dtype=torch.int32)
    counts = slack = None
    if family == "bimodal":
        prompt = _uniform(g, shape, 1, 32)
        short = torch.rand(shape, generator=g, device="cuda") < 0.7
        output = torch.where(short, _uniform(g, shape, 1, 16), _uniform(g, shape, 64, 256))
    elif family == "tiny":
        prompt, output = _uniform(g, shape, 1, 4), _uniform(g, shape, 1, 8)
    elif family in ("online", "robust"):
        prompt, output = _lognormal(g, shape, 512, 1.0, 16, 4096), _lognormal(g, shape, 256, 1.2, 1, 2048)
        if family == "robust":
            slack = (output * torch.rand(shape, generator=g, device="cuda").mul_(0.5)).round_().to(torch.int32)
    elif family == "heavy":
        prompt = _uniform(g, shape, 16, 1024)
        u = torch.rand(shape, generator=g, device="cuda").clamp_(min=1e-7)
        output = u.pow_(-1.0 / 1.5).mul_(8.0).floor_().clamp_(8, 8192).to(torch.int32)
    elif family == "large":
        prompt, output = _lognormal(g, shape, 1024, 1.0, 16, 32768), _lognormal(g, shape, 512, 1.3, 1, 16384)
    else:                                              # profit: accepted requests first, in offer order
        offered = _uniform(g, shape, 1, 1000)
        bucket = (offered + 99) // 100
        accept = (1.0 - offered / ((2 * bucket - 1) * 100.0)).clamp_(min=0.0)
        keep = torch.rand(shape, generator=g, device="cuda") < accept
        counts = keep.sum(1, dtype=torch.int32)
        order = torch.argsort((~keep).to(torch.int32), dim=1, stable=True)
        output = torch.where(keep, offered, 0).gather(1, order).contiguous()
        prompt = torch.zeros_like(output)
    return arrival, prompt, output, counts, slack


def _runs(case):
    pairs = [r.split(":") for r in case["runs"].split(",")]
    return [p for p, _ in pairs], [int(d) for _, d in pairs]


def prepare(case, seed):
    a, p, o, counts, slack = _inputs(case, seed)
    policies, deltas = _runs(case)
    N, n, R = case["instances"], case["n"], len(policies)
    s = {"case": case, "policies": policies, "deltas": deltas}
    flags = sim.FLAG_EPOCH_KERNEL if case["epoch"] else sim.FLAG_STEP_KERNEL
    entry = case["entry"]
    if entry == "noalloc":
        s["flags"] = flags
        s["records"] = torch.empty(R * N * sim.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        s["start"] = torch.empty(R * N * n, dtype=torch.int32, device="cuda")
        s["completion"] = torch.empty(R * N * n, dtype=torch.int32, device="cuda")
    else:
        s["simulator"] = sim.Simulator(N, n, case["B"], C, TAU, P0, epoch=case["epoch"])
    if entry == "host":
        a, p, o, counts, slack = (None if t is None else t.cpu().pin_memory() for t in (a, p, o, counts, slack))
        s["records"] = torch.empty(R * N * sim.RECORD_DTYPE.itemsize, dtype=torch.uint8).pin_memory()
    elif entry == "sweep":
        a, p, o, counts, slack = (None if t is None else t.cpu().numpy() for t in (a, p, o, counts, slack))
    s["inputs"] = (a, p, o, counts, slack)
    return s


def _split(records, case, R):
    """The record bytes as their 16 integer and 8 floating columns (views)."""
    shape = (R, case["instances"], 24)
    return {"integers": records.view(torch.int64).view(shape)[..., :16],
            "costs": records.view(torch.float64).view(shape)[..., 16:]}


def run(s):
    case, policies, deltas = s["case"], s["policies"], s["deltas"]
    a, p, o, counts, slack = s["inputs"]
    R, entry = len(policies), case["entry"]
    if entry == "async":
        rec, st, co = s["simulator"].sweep_async(a, p, o, policies, deltas, case["kv"],
                                                 per_request=case["per_request"], counts=counts, slack=slack)
    elif entry == "sweep":
        res = s["simulator"].sweep(a, p, o, policies, deltas, case["kv"], per_request=True, counts=counts,
                                   slack=slack)
        words = res["records"].view(np.int64).reshape(R, case["instances"], 24)
        return {"integers": words[..., :16], "costs": words.view(np.float64)[..., 16:],
                "start": res["start"], "completion": res["completion"]}
    elif entry == "host":
        status = sim.isjl_sim_run_sweep_host(s["simulator"].handle, policies, deltas, case["kv"], a, p, o,
                                             s["records"], h_count=counts, h_slack=slack)
        if status != sim.ISJL_OK:
            raise sim.IsjlError(status, "isjl_sim_run_sweep_host")
        return _split(s["records"], case, R)
    else:
        rec, st, co = s["records"], s["start"], s["completion"]
        status = sim.isjl_sim_run_sweep_noalloc(case["instances"], case["n"], case["B"], policies, deltas,
                                                case["kv"], a, p, o, rec, st, co, C, TAU, P0, 0, s["flags"],
                                                None, counts, slack)
        if status != sim.ISJL_OK:
            raise sim.IsjlError(status, "isjl_sim_run_sweep_noalloc")
    out = _split(rec, case, R)
    if case["per_request"]:
        shape = (R, case["instances"], case["n"])
        out["start"], out["completion"] = st.view(shape), co.view(shape)
    return out


def work(case):
    """Bytes: each input read once (12 bytes a request, 4 more with slack), each
    output written once (192 bytes a record, 8 bytes a request and run where
    asked for).  Operations: a request's start and its completion each update
    the reservation, the earliest completion, the start range and a counter and
    close an interval of steps (about 12 integer operations each)."""
    R = case["runs"].count(",") + 1
    total = case["instances"] * case["n"]
    per_in = 16 if case["family"] == "robust" else 12
    counts = 4 * case["instances"] if case["family"] == "profit" else 0
    return {"bytes": total * per_in + counts + R * case["instances"] * 192
            + (8 * R * total if case["per_request"] else 0),
            "flops": 24 * R * total}


def tolerance(case):
    """Integers agree bit for bit; the fp64 columns are a handful of operations
    on exact integers, documented to 1e-12 relative."""
    return {"rel": 1e-12, "max": 1e-12, "differ": 0.0}


# ------------------------------------------------- the model, plainly, on the host
def _phase_one(pending, u_sorted, B, alpha, beta):
    """Algorithm 2's Phase ONE over the pending sorted positions: (plan lists per
    worker, long position per worker, d1), or None when it goes to Phase TWO."""
    if len(pending) < 2 or u_sorted[pending[1]] <= alpha:
        return None
    n_long = min(B, sum(1 for p in pending if u_sorted[p] > alpha))
    longs = pending[:n_long]
    del pending[:n_long]
    o1 = u_sorted[longs[0]]
    budget = [0] * B
    for j in range(1, n_long):
        budget[j] = min(2 * alpha, o1 - u_sorted[longs[j]] + beta)
    for j in range(n_long, B):
        budget[j] = alpha
    order = list(range(n_long, B)) + list(range(n_long - 1, 0, -1))   # first fit's worker order
    left = np.array([budget[w] for w in order], dtype=np.int64)
    theta = min(2 * alpha, o1 - u_sorted[longs[-1]] + beta)
    plan = [[] for _ in range(B)]
    sums = [0] * B
    kept = []
    for p in pending:
        o = u_sorted[p]
        fits = np.flatnonzero(left >= o) if o <= theta else ()
        if len(fits) == 0:
            kept.append(p)
            continue
        i = int(fits[0])
        left[i] -= o
        plan[order[i]].append(p)
        sums[order[i]] += o
    pending[:] = kept
    for j in range(n_long):
        plan[j].append(longs[j])
    packs = max([sums[j] for j in range(1, n_long)], default=0)
    return plan, [longs[j] for j in range(n_long)], min(max(packs - alpha, 0), alpha)


def _simulate(policy, delta, B, kv, A, u, o, start, completion):
    """One instance under one run, event by event; returns the record's columns."""
    n = len(o)
    isjl = policy in ("isjl", "isjl_beta")
    alpha = delta
    beta = (math.isqrt(17 * alpha * alpha) - alpha) // 4 if policy == "isjl_beta" else alpha
    order = sorted(range(n), key=lambda i: (-u[i], i))
    u_sorted = [u[i] for i in order]
    pos = [0] * n
    for q, i in enumerate(order):
        pos[i] = q
    pending, queue, head = [], [], 0               # sorted positions; shortest first; arrival order
    running, starts = [], {}                       # heap of (completion, request, worker)
    k = rel = kv_sum = 0
    plan, longs, t0, d1, o1_started, plan_left = [[] for _ in range(B)], [], 0, 0, True, 0
    busy = [False] * B
    W = E = tok = sumc = sumext = maxext = viol = Tb = Tmake = peak_kv = peak_b = 0

    def begin(i, w):
        nonlocal kv_sum, peak_kv, peak_b
        kv_sum += u[i]
        heapq.heappush(running, (k + o[i], i, w))
        starts[i] = k
        busy[w] = True
        start[i], completion[i] = k, k + o[i]
        peak_kv, peak_b = max(peak_kv, kv_sum), max(peak_b, len(running))

    def longest(free):
        for w in free:
            if not pending or kv_sum + u_sorted[pending[0]] > kv:
                return
            begin(order[pending.pop(0)], w)

    done = 0
    while done < n:
        while running and running[0][0] == k:
            c, i, w = heapq.heappop(running)
            kv_sum -= u[i]
            busy[w] = False
            del starts[i]
            done += 1
            sumc += c
            Tmake = c
        while rel < n and A[rel] <= k:
            if policy == "sjf":
                heapq.heappush(queue, (u[rel], rel))
            elif policy != "fcfs":
                bisect.insort(pending, pos[rel])
            rel += 1
        if policy == "fcfs":
            while head < rel and len(running) < B and kv_sum + u[head] <= kv:
                begin(head, busy.index(False))
                head += 1
        elif policy == "sjf":
            while queue and len(running) < B and kv_sum + queue[0][0] <= kv:
                begin(heapq.heappop(queue)[1], busy.index(False))
        elif policy == "ljf":
            if not running:
                longest(range(B))
        else:
            if not running and plan_left == 0 and pending:
                t0, d1, o1_started, longs = k, 0, True, []
                staged = _phase_one(pending, u_sorted, B, alpha, beta)
                if staged:
                    plan, longs, d1 = staged
                    plan_left, o1_started = sum(map(len, plan)), False
            stop = bool(starts) and k - min(starts.values()) > alpha
            if not stop and plan_left:
                for w in range(B):
                    if busy[w] or not plan[w]:
                        continue
                    p = plan[w][0]
                    own = w < len(longs) and p == longs[w]
                    if own and (k < t0 + d1 if w == 0 else not o1_started):
                        continue
                    if kv_sum + u_sorted[p] > kv:
                        stop = True
                        break
                    plan[w].pop(0)
                    plan_left -= 1
                    o1_started = o1_started or (own and w == 0)
                    begin(order[p], w)
            if not stop:
                longest([w for w in range(B) if not busy[w] and not plan[w]])
        if done == n:
            break
        nxt = min([running[0][0]] if running else [INF])
        if rel < n:
            nxt = min(nxt, A[rel])
        if isjl and not o1_started and t0 + d1 > k:
            nxt = min(nxt, t0 + d1)
        if running:
            L, s = nxt - k, len(running)
            s0, s1, total = min(starts.values()), max(starts.values()), sum(starts.values())
            top = L * (k - s0 + 1) + L * (L - 1) // 2          # sum of max r over the steps
            W += s * top
            E += L * (total - s * s0)
            ext = s1 - s0
            sumext += L * ext
            maxext = max(maxext, ext)
            viol += L if ext > delta else 0
            Tb += L
            tok += s * L
        k = nxt
    O, Q = sum(o), sum(x * (x + 1) // 2 for x in o)
    ints = [Tmake, Tb, O, Q, W, E, tok, sumc, sumc - sum(A), sumext, maxext, viol, 0, peak_kv, peak_b, 0]
    c_T, tau_Q, tau_E = C * Tb, TAU * Q, TAU * E
    cost, revenue = (c_T + tau_Q) + tau_E, P0 * O
    return ints, [c_T, tau_Q, tau_E, cost, revenue, revenue - cost, O / Tmake if Tmake else 0.0,
                  sumc / n if n else 0.0]


def exact(case, seed):
    policies, deltas = _runs(case)
    R, N, n = len(policies), case["instances"], case["n"]
    if R * N * n * (1 + case["B"] / 64) > 4e5:         # a plain host simulation takes longer than is useful
        return None
    a, p, o, counts, slack = (None if t is None else t.cpu().numpy() for t in _inputs(case, seed))
    ints, costs = np.zeros((R, N, 16), np.int64), np.zeros((R, N, 8), np.float64)
    st, co = np.full((R, N, n), -1, np.int32), np.full((R, N, n), -1, np.int32)
    for i in range(N):
        m = n if counts is None else int(counts[i])
        length = (p[i, :m] + o[i, :m]).tolist()
        u = length if slack is None else (p[i, :m] + o[i, :m] + slack[i, :m]).tolist()
        for r in range(R):
            ints[r, i], costs[r, i] = _simulate(policies[r], deltas[r], case["B"], case["kv"], a[i, :m].tolist(),
                                                u, length, st[r, i], co[r, i])
    out = {"integers": ints, "costs": costs}
    if case["per_request"]:
        out.update(start=st, completion=co)
    return out
