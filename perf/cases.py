"""Timed cases of the selection library: what a dispatcher built on it has it do.

A case is a plain dict:
  path      which calls one pass makes (see `run`):
              "select"    infaas_select_batch against one load snapshot
              "dispatch"  the same, then infaas_assign_workers for the decided queries
              "step"      infaas_select_batch and infaas_load_update, window after window
              "windows"   infaas_select_update, window after window
              "scale"     the whole control loop of a window: selection, tallies, the autoscaler's
                          decision, the workers, the load advance
              "refresh"   the periodic monitoring tick: one window as in "scale", then the load state
                          read back and states, instances and workers given anew from host tables
  surface   False: `archs` x `hws` x `batches` structured variants per task (archs on hardware
            tiers at power-of-two batch sizes); True: `archs` x `hws` x `batches` variants per task
            drawn on a latency / cost / accuracy trade-off surface (long scan lists)
  tasks, archs, hws, batches      the catalog
  queries, windows                queries per window, windows per pass
  zipf      exponent of the tasks' popularity (0 = uniform)
  mixes     task popularity orders the windows switch between (half of the windows each)
  states    variants carry life-cycle states and loading latencies (state-aware selection)
  queued    initial queue lengths uniform in 0..queued

All results are whole numbers and exact.  Catalog rows come from the package's own generators, the
queries are drawn on the GPU with the same ranges and mixtures.
"""
import math

import numpy as np
import torch

import paper_1905_13348_b200 as P
from paper_1905_13348_b200 import workloads as W

WINDOW_US_PER_QUERY = 40_000 / 65_536        # arrival rate of the workloads: 65,536 queries per 40 ms
SLACK_PCT, LAMBDA_MILLI = 105, 100
WORKERS = 1000


def _case(path, tasks, archs, hws, batches, queries, windows=1, zipf=1.1, surface=False, states=False, queued=0,
          mixes=1, name=None):
    c = {"path": path, "surface": surface, "tasks": tasks, "archs": archs, "hws": hws, "batches": batches,
         "queries": queries, "windows": windows, "zipf": zipf, "mixes": mixes, "states": states, "queued": queued}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a handful of queries that arrived together: latency of one call
        _case("select", 64, 8, 4, 8, 37, name="select_handful"),
        # one application with 32 variants, 10,000 queries
        _case("select", 1, 4, 2, 4, 10_000, zipf=0.0, name="select_small"),
        # 20 applications x 256 variants with standing queues, a million queries, uniform tasks
        _case("select", 20, 8, 4, 8, 1_000_000, zipf=0.0, queued=16, name="select_static_load"),
        # 4 applications x 4096 variants on a trade-off surface: scan lists of several hundred
        _case("select", 4, 64, 8, 8, 1 << 22, zipf=0.0, surface=True, name="select_surface"),
        # replay of a long trace on the largest catalog, with the worker of every query
        _case("dispatch", 128, 16, 4, 8, 65_536_000, zipf=1.5, name="dispatch_trace"),
        # the benchmark's step: 2^24 queries decided, then their load folded back (twice per pass,
        # so that the second batch is decided against the load of the first)
        _case("step", 64, 8, 4, 8, 1 << 24, windows=2, name="step_batch"),
        # mid-size windows of an odd length, closed by one call each
        _case("windows", 48, 8, 3, 8, 1_500_007, windows=4, name="windows_mid"),
        # a live stream: windows of 65,536 queries, load refreshed after each
        _case("windows", 64, 8, 4, 8, 65_536, windows=16, name="windows_stream"),
        # the same on twice the tasks and variants with a task mix that switches
        _case("windows", 128, 16, 4, 8, 65_536, windows=16, zipf=1.5, mixes=2, name="windows_switching"),
        # small odd windows on long lists: the load update of large tasks
        _case("windows", 4, 64, 8, 8, 20_011, windows=4, zipf=0.0, surface=True, name="windows_surface"),
        # the control loop with life-cycle states: autoscaler and worker choice in every window
        _case("scale", 64, 8, 4, 8, 65_536, windows=8, states=True, name="scale_states"),
        # a monitoring tick
        _case("refresh", 64, 8, 4, 8, 65_536, states=True, name="refresh_tick"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    path = rng.choice(["select", "select", "dispatch", "step", "step", "windows", "windows", "windows", "scale",
                       "refresh"])
    surface = path in ("select", "step", "windows") and rng.random() < 0.15
    if surface:
        tasks, archs, hws, batches = rng.randint(1, 4), rng.randint(16, 64), 8, rng.randint(4, 8)
    else:
        tasks, archs, hws, batches = _log_int(rng, 1, 128), rng.randint(1, 16), rng.randint(1, 4), rng.randint(1, 8)
    if path in ("select", "dispatch"):
        queries, windows = _log_int(rng, 1, 1 << 25), 1
    elif path == "step":
        queries, windows = _log_int(rng, 1000, 1 << 24), 2
    elif path == "windows":
        queries, windows = _log_int(rng, 1000, 1 << 21), rng.randint(2, 16)
    else:
        queries, windows = _log_int(rng, 1000, 1 << 18), rng.randint(2, 8) if path == "scale" else 1
    if surface:
        queries = min(queries, 1 << 22)
    return _case(path, tasks, archs, hws, batches, queries, windows,
                 zipf=0.0 if surface else rng.choice([0.0, 1.1, 1.5]), surface=surface,
                 states=path in ("scale", "refresh") or (not surface and rng.random() < 0.25),
                 queued=rng.choice([0, 0, 16]), mixes=rng.choice([1, 2]) if windows > 1 else 1)


def _variants(case):
    return case["tasks"] * case["archs"] * case["hws"] * case["batches"]


def _rows(case, rng):
    T, per_task = case["tasks"], case["archs"] * case["hws"] * case["batches"]
    if case["surface"]:
        rows = W.tradeoff_catalog(rng, T, per_task)
        if case["queued"]:
            rows["queued"] = rng.integers(0, case["queued"] + 1, rows.size)
        return rows
    return W.structured_catalog(rng, T, case["archs"], case["hws"], [1 << b for b in range(case["batches"])],
                                queued_hi=case["queued"])


def _u16(t):
    """int64 values 0..65535 as the 16-bit array the library reads."""
    return (t - ((t >> 15) << 16)).to(torch.int16)


class _Queries:
    """Draws windows of queries on the GPU."""

    def __init__(self, case, rows, seed):
        self.case, self.dev = case, torch.device("cuda")
        self.gen = torch.Generator(self.dev).manual_seed(int(seed))
        T = case["tasks"]
        pmf = W._zipf_pmf(T, case["zipf"])
        self.cdf = torch.from_numpy(np.cumsum(pmf).clip(0, 1).astype(np.float32)).to(self.dev)
        self.cdf[-1] = 1.0
        self.perms = [torch.randperm(T, generator=self.gen, device=self.dev) for _ in range(case["mixes"])]
        order = np.lexsort((rows["acc_bp"], rows["task"]))
        acc = rows["acc_bp"][order].astype(np.int64).reshape(T, -1)      # every task has the same number of variants
        lat = rows["lat_us"][np.lexsort((rows["lat_us"], rows["task"]))].astype(np.int64).reshape(T, -1)
        self.acc, self.lat = torch.from_numpy(acc).to(self.dev), torch.from_numpy(lat).to(self.dev)

    def window(self, k):
        """(task u16, slo u32, min_acc u16) of the k-th window."""
        n, T = self.case["queries"], self.case["tasks"]
        parts, CH = [], 1 << 24
        perm = self.perms[k * len(self.perms) // self.case["windows"]]
        for lo in range(0, n, CH):
            m = min(CH, n - lo)
            u = torch.rand(3, m, generator=self.gen, device=self.dev)
            t = perm[torch.searchsorted(self.cdf, u[0], right=True).clamp_(max=T - 1)]
            V = self.acc.shape[1]
            if self.case["surface"]:
                # requirements from the task's own attribute quantiles, about a tenth infeasible
                slo = self.lat[t, (u[1] * V).long().clamp_(max=V - 1)]
                ma = self.acc[t, (u[2] * W.C4_ACC_QUANTILE_SCALE * V).long().clamp_(max=V - 1)]
            else:
                # SLO log-uniform over 1 ms .. 1 s; 30 % of the accuracies above the task's median
                slo = torch.exp(math.log(1000.0) + u[1] * (math.log(1_000_001.0) - math.log(1000.0))).long()
                slo.clamp_(1000, 1_000_000)
                above = u[2] < 0.3
                f = torch.where(above, u[2] / 0.3, (u[2] - 0.3) / 0.7)
                amin, amed, amax = self.acc[:, 0][t], self.acc[:, (V - 1) // 2][t], self.acc[:, -1][t]
                a_lo = torch.where(above, amed + 1, amin)
                a_hi = torch.where(above, torch.maximum(amax, amed + 1), amed)
                ma = a_lo + (f * (a_hi - a_lo + 1)).long().clamp_(min=0)
                ma = torch.minimum(ma, a_hi)
            parts.append((_u16(t), slo.to(torch.int32), _u16(ma)))
        return tuple(torch.cat([p[i] for p in parts]) if len(parts) > 1 else parts[0][i] for i in range(3))


def _worker_tables(rng, rows):
    """Half of the variants loaded on one to three of the workers."""
    nv = rows.size
    loaded = np.flatnonzero(rng.random(nv) < 0.5)
    iv = np.repeat(loaded, rng.integers(1, 4, loaded.size)).astype(np.uint32)
    return (iv, rng.integers(0, WORKERS, iv.size).astype(np.uint32), rng.integers(0, 10_000, iv.size).astype(np.uint32),
            rng.integers(0, 4, WORKERS).astype(np.uint8), rng.integers(0, 10_000, WORKERS).astype(np.uint32))


def prepare(case, seed):
    """The catalog handle with its tables, the windows' queries on the GPU, and the output arrays."""
    rng = np.random.Generator(np.random.PCG64([int(seed), 11]))
    rows = _rows(case, rng)
    T, nv, n = case["tasks"], rows.size, case["queries"]
    cat = P.infaas_catalog_load(rows, T, torch.cuda.current_device())
    s = {"case": case, "cat": cat, "window_us": max(1, int(round(n * WINDOW_US_PER_QUERY)))}
    q = _Queries(case, rows, seed)
    s["queries"] = [q.window(k) for k in range(case["windows"])]
    i32 = dict(dtype=torch.int32, device="cuda")
    s["decision"] = [torch.empty(n, **i32) for _ in range(case["windows"])]
    path = case["path"]
    if path in ("dispatch", "scale", "refresh"):
        s["worker"] = [torch.empty(n, **i32) for _ in range(case["windows"])]
        s["workers"] = _worker_tables(rng, rows)
        P.infaas_workers_config(cat, *s["workers"])
    if path in ("scale", "refresh"):
        # one instance of the variants that are loaded, SLOs around the middle of the queries'
        inst = (rng.random(nv) < 0.1).astype(np.uint32)
        s["autoscale"] = (inst, rng.integers(20_000, 200_000, T).astype(np.uint32))
        P.infaas_autoscale_config(cat, *s["autoscale"])
        s["actions"] = [(torch.empty(T, **i32), torch.empty(T, **i32)) for _ in range(case["windows"])]
    if case["states"]:
        s["states"] = W.variant_states(nv, seed=int(seed))
        P.infaas_catalog_set_states(cat, *s["states"])
    return s


def run(s):
    cat, path, wus = s["cat"], s["case"]["path"], s["window_us"]
    out = {"decision": s["decision"]}
    for k, (task, slo, min_acc) in enumerate(s["queries"]):
        d = s["decision"][k]
        if path == "windows":
            P.infaas_select_update(cat, task, slo, min_acc, d, wus)
            continue
        P.infaas_select_batch(cat, task, slo, min_acc, d)
        if path == "step":
            P.infaas_load_update(cat, d, wus)
        elif path == "dispatch":
            P.infaas_assign_workers(cat, d, s["worker"][k])
        elif path in ("scale", "refresh"):
            P.infaas_tally(cat, d)
            P.infaas_autoscale_step(cat, wus, SLACK_PCT, LAMBDA_MILLI, *s["actions"][k])
            P.infaas_assign_workers(cat, d, s["worker"][k])
            P.infaas_advance(cat, wus)
    if path == "refresh":
        out["load"] = P.infaas_catalog_get_state(cat)
        out["state"] = P.infaas_catalog_get_states(cat)
        P.infaas_catalog_set_states(cat, *s["states"])
        P.infaas_autoscale_config(cat, *s["autoscale"])
        P.infaas_workers_config(cat, *s["workers"])
    if "worker" in s:
        out["worker"] = s["worker"]
    if "actions" in s:
        out["actions"] = s["actions"]
    return out


def work(case):
    """8 B of every query read and its 4 B decision written, 4 B more where the worker is wanted; the
    catalog's rows (24 B, those of the tasks that can be asked for) read once; an update reads and
    writes queue, latency and total of every variant."""
    n, w, nv, path = case["queries"], case["windows"], _variants(case), case["path"]
    b = n * w * (16 if path in ("dispatch", "scale", "refresh") else 12)
    b += 24 * nv * min(case["tasks"], n * w) // case["tasks"]
    if path not in ("select", "dispatch"):
        b += w * nv * 28
    if path in ("scale", "refresh"):
        b += w * nv * 12 + w * case["tasks"] * 12          # throughput and instances in, actions out
    if path == "refresh":
        b += nv * (16 + 1 + 5 + 4) + nv * 12               # state out, tables in
    return {"bytes": b, "flops": 0}


def tolerance(case):
    return "exact"
