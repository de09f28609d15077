"""Performance cases: what a user of the scheduler simulation runs through its
public entry points, from one window's alpha sweep to a grid over long traces.

A case is a dict of plain values:

  path     how the program calls the library
           "window"  `tuner.gpu_backend`: a handle of its own for one window's
                     sweep over alpha (create, run, results, per-call log, destroy)
           "static"  `hxsim.run_static`: one trace, nothing allocated
           "handle"  a kept `hxsim.Sim` whose traces are resident: run, results, best
           "refresh" a kept `hxsim.Sim` given new traces first: upload, run, results, best
  recipe   a recipe of `workloads` (index as text, or a key of `workloads.EXTRA`):
           arrivals, token lengths, cluster, grid
  traces, queries   traces and queries per trace
  points   grid points, spread evenly over the recipe's grid (0: all of it);
           with "window" the number of alpha values
  mixed    True: the points take the four scheduler pairs of the evaluation's
           baselines and ablations in turn (round robin with FCFS or urgency
           queues, balanced dispatch with FCFS or least-laxity queues)
"""
import heapq
import math

import numpy as np
import torch

from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import tuner as T
from paper_2505_05286_gb300 import workloads as W

FIELDS = ("p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status")
PAIRS = ((W.DISPATCH_RR, W.POLICY_FCFS), (W.DISPATCH_RR, W.POLICY_PQ), (W.DISPATCH_WB, W.POLICY_FCFS),
         (W.DISPATCH_WB, W.POLICY_LLF))
MOST_EVENTS = 1.25e9  # simulated calls of the largest case


def _case(name, path, recipe, traces, queries, points=0, mixed=False):
    c = dict(path=path, recipe=recipe, traces=traces, queries=queries, points=points, mixed=mixed)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the online tuner of a small deployment: 100 s at 2 queries/s, alpha = 0, 0.1, ..., 1
        _case("window-200q", "window", "0", 1, 200, 11),
        # the same for 64 instances: 150 s at 20 queries/s
        _case("window-3000q-64inst", "window", "4", 1, 3000, 11),
        # a caller that may not allocate: one window over a 4 x 4 grid
        _case("static-200q", "static", "0", 1, 200),
        # eight new windows of agentic queries (~20 calls each) on a kept handle
        _case("refresh-agentic", "refresh", "paper-shaped", 8, 400),
        # a day of many long windows on a kept handle: upload and preparation weigh most
        _case("refresh-64x3001q", "refresh", "3", 64, 3001, 16),
        # an evening's traces over a coarse grid: fewer simulations than the GPU has warps
        _case("small-sweep", "handle", "1", 8, 2000),
        # bursty arrivals, 2 to 8 candidates, 256 points
        _case("bursty", "handle", "2", 32, 5000),
        # heavy-tailed lengths on 32 instances of four types, an odd number of traces
        _case("hetero-19x5003q", "handle", "3", 19, 5003),
        # the largest cluster and grid over full-length traces
        _case("ceiling-8x20000q", "handle", "4", 8, 20000),
        # the baselines and ablations of the evaluation side by side
        _case("policies-64inst", "handle", "4", 10, 6001, 256, True),
        # two tenants, workflow queries against single-shot requests: per-tenant results
        _case("competing-tenants", "handle", "competing-25", 24, 2000),
        # instances that slow down or stop, with timeouts and re-issue
        _case("faulty", "handle", "faulty", 24, 2000),
    ]


def _recipe(case):
    r = case["recipe"]
    return (W.RECIPES[int(r)], int(r)) if r.isdigit() else (W.EXTRA[r], W.EXTRA_ID[r])


def _calls_per_query(recipe):
    k = sum(recipe.k_range) / 2
    fix = sum(recipe.p_err ** j for j in range(1, recipe.rmax + 1))
    return (2 + k * (1 + fix)) * (1 + recipe.single_frac)


def _n_points(case):
    if case["points"]:
        return case["points"]
    return W.make_grid(_recipe(case)[0]).n_points


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    path = rng.choice(("window", "static", "refresh", "handle", "handle", "handle"))
    mixed = False
    if path == "window":
        recipe = rng.choice(("0", "1", "2", "3", "4"))
        traces, queries, points = 1, _log(rng, 5, 4000), rng.choice((1, 11, 11, 21))
    elif path == "static":
        recipe = rng.choice(("0", "1", "2", "competing-25"))
        traces, queries, points = 1, _log(rng, 20, 1500), _log(rng, 1, 64 if recipe != "0" else 16)
    elif path == "refresh":
        recipe = rng.choice(("1", "2", "3", "paper-shaped", "two-tenant"))
        traces, queries, points = _log(rng, 1, 64), _log(rng, 50, 4000), _log(rng, 1, 16)
    else:
        recipe = rng.choice(("1", "2", "3", "4", "noisy-estimate", "two-tenant", "competing-50", "faulty"))
        traces, queries = _log(rng, 1, 32), _log(rng, 1400 if recipe == "faulty" else 100, 12000)
        mixed = rng.random() < 0.25
        full = W.make_grid(W.RECIPES[int(recipe)] if recipe.isdigit() else W.EXTRA[recipe]).n_points
        points = _log(rng, 4, full)
    case = _case(None, path, recipe, traces, queries, points, mixed)
    per_trace = queries * _calls_per_query(_recipe(case)[0]) * points
    case["traces"] = max(1, min(traces, int(0.6 * MOST_EVENTS / per_trace)))
    return case


def _grid(case, recipe):
    g = W.make_grid(recipe)
    n = case["points"]
    if n and n < g.n_points:
        g = W.subset_grid(g, [int(i * (g.n_points - 1) / max(1, n - 1) + 0.5) for i in range(n)])
    if case["mixed"]:
        pair = [PAIRS[p % 4] for p in range(g.n_points)]
        g.dispatch_policy = np.array([d for d, _ in pair], np.uint8)
        g.local_policy = np.array([q for _, q in pair], np.uint8)
    return g


def _inputs(case, seed):
    recipe, rid = _recipe(case)
    traces = [W.make_trace(recipe, rid, 1024 * (seed + 1) + t, case["queries"]) for t in range(case["traces"])]
    cluster = W.make_cluster(recipe)
    if case["path"] == "window":
        n = case["points"]
        alphas = [i * W.SCALE // max(1, n - 1) for i in range(n)]
        grid = T.OnlineTuner(cluster, alphas_fp=alphas, beta_us2=recipe.c_ref_us ** 2).grid_of(alphas)
    else:
        grid = _grid(case, recipe)
    return recipe, traces, cluster, grid


def prepare(case, seed):
    recipe, traces, cluster, grid = _inputs(case, seed)
    state = dict(path=case["path"], traces=traces, cluster=cluster, grid=grid, objective=recipe.objective,
                 tenants=cluster.n_tenants > 1 or cluster.faults is not None)
    if case["path"] in ("handle", "refresh"):
        state["sim"] = H.Sim(traces, cluster, grid)
    return state


def _table(res):
    """Every field of the results but the clock diagnostic, which varies from run to run."""
    out = {f: np.ascontiguousarray(res[f]) for f in FIELDS}
    out["digest"] = out["digest"].view(np.int64)
    return out


def run(state):
    path = state["path"]
    if path == "window":
        res, latency = T.gpu_backend(state["traces"][0], state["cluster"], state["grid"])
        return dict(_table(res), latency=latency)
    if path == "static":
        res, best = H.run_static(state["traces"][0], state["cluster"], state["grid"], state["objective"])
        return dict(_table(res), best=np.array(best, np.int64))
    sim = state["sim"]
    if path == "refresh":
        sim.upload(state["traces"])
    sim.run(torch.cuda.current_stream())
    out = _table(sim.results())
    point, sum_p95, slo, per_trace = sim.best(state["objective"])
    out["best"] = np.array((point, sum_p95, slo), np.int64)
    out["per_trace"] = per_trace
    if state["tenants"]:
        extra = sim.extras()
        for f in ("slo_met", "n_done", "reissued", "p95_us"):
            out["tenant_" + f] = np.ascontiguousarray(extra[f])
    return out


def work(case):
    """Bytes: every trace, cluster and grid array once and every result once.
    Operations, per simulated call: two reward divisions and one budget
    division (about 10 each), a score and a comparison per instance type, one
    path each through a tree of the instances' rewards and one of their next
    completions, and about 30 for the queue, the slots and the digest."""
    recipe, _ = _recipe(case)
    points = _n_points(case)
    calls = case["traces"] * case["queries"] * _calls_per_query(recipe)
    per_call = 3 * 10 + 3 * len(recipe.types) + 2 * math.ceil(math.log2(sum(recipe.inst_counts))) + 30
    return {"bytes": calls * 15 + case["traces"] * case["queries"] * 14 + points * 30 + case["traces"] * points * 48,
            "flops": calls * points * per_call}


def tolerance(case):
    # int64 microseconds and fixed point throughout: every value is determined
    return "exact"


# ----------------------------------------------------------------------------
# The same simulation in plain Python integers
# ----------------------------------------------------------------------------
_M64 = (1 << 64) - 1


def _mix(t, tag):
    z = ((t * 0x9E3779B97F4A7C15) & _M64) ^ tag
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _trunc(a, b):
    return a // b if a >= 0 else -(-a // b)


def _p95(latencies):
    s = sorted(latencies)
    return s[(95 * len(s) + 99) // 100 - 1] if s else 0


def _simulate(trace, cluster, grid, p):
    """One (trace, point) pair: the result row, the tenants' row and the query latencies."""
    pre, dec = cluster.prefill_tok_s.tolist(), cluster.decode_us_tok.tolist()
    ty = cluster.inst_type.tolist()
    n_inst, n_types = len(ty), len(pre)
    slots = [int(cluster.slots[t]) for t in ty]
    count = [ty.count(t) for t in range(n_types)]
    A, G, beta = int(grid.alpha_fp[p]), int(grid.gamma_fp[p]), int(grid.beta_us2[p])
    rho, rmax = int(grid.rho[p]), int(cluster.rmax)
    local, balanced = int(grid.local_policy[p]), int(grid.dispatch_policy[p]) == W.DISPATCH_WB

    def cost(t, prompt, out):
        return -(-prompt * 1_000_000 // pre[t]) + out * dec[t]

    prompt, out, believed = trace.prompt.tolist(), trace.out.tolist(), trace.out_est.tolist()
    stage, cand, retry = trace.stage.tolist(), trace.cand.tolist(), trace.retry.tolist()
    base, arrival, ks = trace.call_base.tolist(), trace.arrival_us.tolist(), trace.k.tolist()
    tenant = trace.tenant.tolist() if trace.tenant is not None else [0] * len(ks)
    nq, nc = len(arrival), len(prompt)
    mult = [int(cluster.slo_mult_fp)] * 4
    if cluster.tenant_slo_mult_fp is not None:
        mult[:len(cluster.tenant_slo_mult_fp)] = [int(x) for x in cluster.tenant_slo_mult_fp]
    est = [[cost(t, prompt[j], believed[j]) for t in range(n_types)] for j in range(nc)]
    svc = [[cost(t, prompt[j], out[j]) for t in range(n_types)] for j in range(nc)]
    tbar = [sum(c * e for c, e in zip(count, est[j])) // n_inst for j in range(nc)]
    sref, oref = cluster.stage_ref_prompt.tolist(), cluster.stage_ref_out.tolist()
    cref = [sum(count[t] * cost(t, sref[s], oref[s]) for t in range(n_types)) // n_inst for s in range(4)]

    query, after, rest, deadline = [0] * nc, [None] * nc, [0] * nc, [0] * nq
    for i in range(nq):
        b, e = base[i], base[i + 1]
        chain, first = {}, 0
        for j in range(b, e):
            query[j] = i
            ref = cost(cluster.ref_type, prompt[j], out[j])
            if stage[j] in (W.STAGE_G, W.STAGE_C):
                chain[cand[j]] = chain.get(cand[j], 0) + ref
                u = retry[j]
                rest[j] = min(rho, rmax - u) * cref[2] + cref[3]
                nxt = [c for c in range(b, e) if stage[c] == W.STAGE_C and cand[c] == cand[j] and retry[c] == u + 1]
                after[j] = nxt[0] if nxt else None
            else:
                first += ref
                if stage[j] == W.STAGE_S:
                    rest[j] = cref[1] + min(rho, rmax) * cref[2] + cref[3]
        exclusive = first + max(chain.values(), default=0)
        deadline[i] = arrival[i] + mult[tenant[i]] * exclusive // W.SCALE

    queue_us, running, waiting = [0] * n_inst, [[] for _ in ty], [[] for _ in ty]
    heads, left, digest, rr, reissued = [], list(ks), 0, 0, 0
    latency, done, slo, done_t, slo_t, lat_t = [0] * nq, 0, 0, [0] * 4, [0] * 4, [[], [], [], []]
    events = makespan = now = qa = 0
    faults = [] if cluster.faults is None else [tuple(int(f[x]) for x in ("inst", "t0_us", "t1_us", "slow_fp"))
                                                for f in cluster.faults]
    while True:
        while heads and (not running[heads[0][1]] or running[heads[0][1]][0][:2] != (heads[0][0], heads[0][2])):
            heapq.heappop(heads)  # an entry that is not its instance's next completion any more
        if not heads and qa == nq:
            break
        released, avoid, touched = [], -1, set()
        if heads and (qa == nq or heads[0][0] <= arrival[qa]):
            now, m, _ = heapq.heappop(heads)
            _, j, failed = heapq.heappop(running[m])
            if running[m]:
                heapq.heappush(heads, (running[m][0][0], m, running[m][0][1]))
            touched.add(m)
            queue_us[m] -= est[j][ty[m]]
            i = query[j]
            if failed:
                reissued += 1
                released, avoid = [j], m if n_inst > 1 else -1
            else:
                events += 1
                if stage[j] == W.STAGE_S:
                    released = list(range(j + 1, j + 1 + ks[i]))
                elif stage[j] == W.STAGE_E:
                    latency[i] = now - arrival[i]
                    done, makespan, u = done + 1, now, tenant[i]
                    slo, slo_t[u], done_t[u] = slo + (now <= deadline[i]), slo_t[u] + (now <= deadline[i]), done_t[u] + 1
                    lat_t[u].append(latency[i])
                    digest += _mix(now, (i << 8) | 0xFF)
                elif after[j] is not None:
                    released = [after[j]]
                else:
                    left[i] -= 1
                    if left[i] == 0:
                        released = [base[i + 1] - 1]
        else:
            now, released, qa = arrival[qa], [base[qa]], qa + 1
        for j in released:
            if balanced:
                best, m = None, -1
                for c in range(n_inst):
                    if c != avoid:
                        s = (W.SCALE - A) * min(beta // max(queue_us[c], 1), 2 ** 43 - 1) - A * est[j][ty[c]]
                        if best is None or s > best:
                            best, m = s, c
            else:
                m = rr if rr != avoid else (rr + 1) % n_inst
                rr = (m + 1) % n_inst
            avoid = -1
            e = est[j][ty[m]]
            queue_us[m] += e
            path_us = tbar[j] + rest[j]
            if local == W.POLICY_PQ:
                key = -(W.SCALE * (e - _trunc((deadline[query[j]] - now) * tbar[j], path_us)) - G * now)
            else:
                key = now if local == W.POLICY_FCFS else deadline[query[j]] - path_us
            heapq.heappush(waiting[m], (key, j))
            touched.add(m)
        for m in sorted(touched):
            while waiting[m] and len(running[m]) < slots[m]:
                j = heapq.heappop(waiting[m])[1]
                span, failed = svc[j][ty[m]], False
                for f, t0, t1, slow in faults:
                    if f == m and t0 <= now < t1:
                        limit = est[j][ty[m]] * cluster.timeout_mult_fp // W.SCALE
                        span = -(-span * slow // W.SCALE)
                        if cluster.timeout_mult_fp > 0 and (slow == 0 or span > limit):
                            span, failed = limit, True
                        break
                heapq.heappush(running[m], (now + span, j, failed))
                if running[m][0][1] == j:
                    heapq.heappush(heads, (now + span, m, j))
                digest += _mix(now, (j << 8) | m)
    row = (_p95(latency), makespan, events, digest & _M64, slo, done, 0)
    return row, (slo_t, done_t, reissued, [_p95(v) for v in lat_t]), latency


def _best(rows, n_points, queries, objective):
    """The best point of a table of (sum P95, SLO hits) pairs, and its sums."""
    def order(p):
        p95, slo = rows[p]
        if objective == W.OBJ_P95_SLO95:
            return (0, p95, p) if slo * 100 >= 95 * queries else (1, -slo, p95, p)
        return (p95, p)
    p = min(range(n_points), key=order)
    return (p, *rows[p])


def exact(case, seed):
    recipe, _ = _recipe(case)
    calls = case["traces"] * case["queries"] * _calls_per_query(recipe)
    if calls * _n_points(case) * (10 + 0.5 * sum(recipe.inst_counts)) > 14e6:  # about 15 s
        return None
    recipe, traces, cluster, grid = _inputs(case, seed)
    P = grid.n_points
    sims = [_simulate(t, cluster, grid, p) for t in traces for p in range(P)]
    out = {f: np.array([s[0][i] for s in sims], np.uint64 if f == "digest" else np.int64) for i, f in enumerate(FIELDS)}
    out["digest"] = out["digest"].view(np.int64)
    if case["path"] == "window":
        return dict(out, latency=np.array(sims[0][2], np.int64))
    pairs = [(s[0][0], s[0][4]) for s in sims]
    total = [tuple(sum(pairs[t * P + p][i] for t in range(len(traces))) for i in (0, 1)) for p in range(P)]
    nq = [t.n_queries for t in traces]
    out["best"] = np.array(_best(total, P, sum(nq), recipe.objective), np.int64)
    if case["path"] == "static":
        return out
    out["per_trace"] = np.array([_best(pairs[t * P:(t + 1) * P], P, nq[t], recipe.objective)[0]
                                 for t in range(len(traces))], np.int64)
    if cluster.n_tenants > 1 or cluster.faults is not None:
        for i, f in enumerate(("slo_met", "n_done", "reissued", "p95_us")):
            out["tenant_" + f] = np.array([s[1][i] for s in sims], np.int64)
    return out
