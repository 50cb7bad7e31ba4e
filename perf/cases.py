"""What users of this framework have it do, as cases that can be timed.

A case is one call (or the few calls that belong together) of the public entry points in
`paper_2008_12260_b200.api`, at a size drawn from the ranges this repository's own configurations
span: the 8-job "tiny" cluster, the 64-GPU testbed of the paper, the 160-job trace, the 2048-GPU
"large" cluster and the 8192-job "stress" population.  Kinds:

  round       schedule_round / schedule_round_host: a scheduling round of Sec. 4.3 from the job
              parameters to the best allocation (what the scheduler runs every 60 seconds)
  table       build_speedup_table / build_speedup_table_msample: the tables of Eq. 13 and 15 alone
              (a simulator or an auto-scaler asks for these without a search)
  generation  ga_generation + eval_fitness on dense matrices: one step of a search that the caller
              drives (as `dist.evolve_sharded` does), all candidates on this GPU
  fitness     eval_fitness / eval_fitness_racks of a population the caller brings
  fit         fit_throughput_model: the profiled iteration times of many jobs (Sec. 4.1)

Inputs come from `paper_2008_12260_b200.synth` (job parameters, allocations, populations) and from
the seed alone.
"""
import math

import numpy as np
import torch

from paper_2008_12260_b200 import api, synth

GPU = "cuda"
_streams = []


def _stream():
    """The program's stream: one for all that it asks of this GPU (not the default stream, on which
    rounds do not replay as graphs)."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


# Rounds.  nodes x gpus, jobs (rows of the matrices), the (m, s) grid, population and generations;
# `active`: share of the jobs that are in the cluster at the moment (a trace keeps a row for every
# job it will ever see); `host`: job arrays and matrices in pinned host memory, as a scheduler
# process has them; `racks`: the cluster is split into that many racks (0: one).
ROUND = {"kind": "round", "nodes": 16, "gpus": 4, "jobs": 48, "grid_m": 64, "grid_s": 16, "population": 100,
         "generations": 100, "elite": 4, "mutate": 0.08, "init": 0.25, "active": 1.0, "host": False, "racks": 0}
TABLE = {"kind": "table", "nodes": 256, "gpus": 8, "jobs": 1024, "grid_m": 128, "grid_s": 32, "samples": 0}
GENERATION = {"kind": "generation", "nodes": 256, "gpus": 8, "jobs": 1024, "population": 512, "elite": 16,
              "mutate": 0.01, "init": 0.02}
FITNESS = {"kind": "fitness", "nodes": 2048, "gpus": 8, "jobs": 8192, "count": 64, "p": -1.0, "penalty": False,
           "racks": 0}
FIT = {"kind": "fit", "jobs": 1024, "observations": 64}


def _case(base, **kw):
    c = dict(base)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest round anyone runs: a four-node cluster (launches and host time are what it costs)
        _case(ROUND, name="round_tiny", nodes=4, jobs=8, grid_m=32, grid_s=8, population=32, generations=10, elite=2,
              mutate=0.2),
        # the paper's own cluster: 16 nodes x 4 GPUs, arrays already on the GPU
        _case(ROUND, name="round_testbed"),
        # the scheduler of a running trace: 160 rows of which a quarter is active, arrays on the host
        _case(ROUND, name="round_trace_host", jobs=160, active=0.25, host=True),
        # a middling cluster whose node count is no multiple of anything
        _case(ROUND, name="round_ragged", nodes=75, gpus=8, jobs=210, grid_m=50, population=150, generations=100,
              elite=6, mutate=0.04),
        # the testbed grown to four racks with the third synchronisation pair
        _case(ROUND, name="round_racks", nodes=32, jobs=96, racks=4),
        # the largest cluster, end to end from host memory: what the headline of the benchmark measures
        _case(ROUND, name="round_large_host", nodes=256, gpus=8, jobs=1024, grid_m=128, grid_s=32, population=512,
              generations=200, elite=16, mutate=0.01, init=0.02, host=True),
        # tables alone, all three outputs, for the largest cluster
        _case(TABLE, name="table_large"),
        # tables by sampling total batch sizes, for a trace's jobs
        _case(TABLE, name="table_samples", nodes=16, gpus=4, jobs=160, grid_m=1, grid_s=1, samples=128),
        # a caller-driven search on dense matrices, largest cluster
        _case(GENERATION, name="generation_large"),
        # a large population of mostly empty matrices, evaluated as fast as they can be read
        _case(FITNESS, name="fitness_stress"),
        # an odd-sized population with the re-allocation penalty and another exponent
        _case(FITNESS, name="fitness_ragged", nodes=251, jobs=777, count=300, p=0.5, penalty=True),
        # all agents' throughput models refitted at once
        _case(FIT, name="fit_agents"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round", "round", "round", "table", "generation", "fitness", "fit"])
    if kind == "round":
        while True:
            c = _case(ROUND, nodes=_log_int(rng, 4, 256), gpus=rng.choice([2, 4, 8]), jobs=_log_int(rng, 8, 1024),
                      grid_m=rng.randint(32, 128), grid_s=rng.randint(8, 32), population=_log_int(rng, 32, 512),
                      generations=_log_int(rng, 10, 200), elite=rng.randint(0, 16), mutate=rng.uniform(0.01, 0.2),
                      init=rng.uniform(0.02, 0.3), active=rng.choice([1.0, 1.0, 0.5, 0.25]),
                      host=rng.random() < 0.5, racks=rng.choice([0, 0, 0, 0, 4]))
            # a tenth of the largest round's matrices: odd sizes and racks do more work for each entry
            if c["population"] * c["jobs"] * c["nodes"] * c["generations"] <= 0.1 * 512 * 1024 * 256 * 200:
                return c
    if kind == "table":
        return _case(TABLE, nodes=_log_int(rng, 4, 256), gpus=rng.choice([2, 4, 8]), jobs=_log_int(rng, 8, 1024),
                     grid_m=rng.randint(32, 128), grid_s=rng.randint(8, 32),
                     samples=rng.choice([0, 0, rng.randint(32, 128)]))
    if kind == "generation":
        while True:
            c = _case(GENERATION, nodes=_log_int(rng, 8, 256), gpus=rng.choice([4, 8]), jobs=_log_int(rng, 16, 1024),
                      population=_log_int(rng, 32, 512), elite=rng.randint(0, 16), mutate=rng.uniform(0.01, 0.1),
                      init=rng.uniform(0.02, 0.3))
            if c["population"] * c["jobs"] * c["nodes"] <= 0.25 * 512 * 1024 * 256:
                return c
    if kind == "fitness":
        while True:
            c = _case(FITNESS, nodes=_log_int(rng, 8, 2048), jobs=_log_int(rng, 16, 8192), count=_log_int(rng, 32, 512),
                      p=rng.choice([-1.0, 0.5, 1.0, 0.0, -10.0]), penalty=rng.random() < 0.5,
                      racks=rng.choice([0, 0, 0, 8]))
            if c["count"] * c["jobs"] * c["nodes"] <= (0.25 if c["racks"] else 1.0) * 64 * 8192 * 2048:
                return c
    return _case(FIT, jobs=_log_int(rng, 16, 1024), observations=_log_int(rng, 16, 128))


# ---- inputs ------------------------------------------------------------------------------------
def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(GPU)


def _jobs(case, cluster, seed):
    rng = np.random.default_rng(seed)
    jobs = synth.draw_jobs(case["jobs"], seed, case.get("grid_m", 1), max(case.get("grid_s", 8), 8), cluster.k_max, phi_hi=1e6,
                           with_history=True)
    if case.get("active", 1.0) < 1.0:
        jobs.active = (rng.random(case["jobs"]) < case["active"]).astype(np.uint8)
        jobs.active[int(rng.integers(case["jobs"]))] = 1
    fk, fn = api.fair_share(cluster.node_capacity, int(jobs.active.sum()), cluster.k_max)
    jobs.fair_k = np.full(case["jobs"], fk, np.int32)
    jobs.fair_n = np.full(case["jobs"], fn, np.int32)
    return jobs


def _scheduler(case, cluster, stream, seed):
    return api.Scheduler(
        node_capacity=cluster.node_capacity, num_jobs=case["jobs"], grid_m=case.get("grid_m", 1),
        grid_s=case.get("grid_s", 1), population=case.get("population", 1), p=case.get("p", -1.0),
        thr_mutate=synth.prob_to_threshold(case.get("mutate", 0.0)), thr_init=synth.prob_to_threshold(case.get("init", 0.0)),
        num_elite=case.get("elite", 0), seed=seed, stream=stream.cuda_stream)


def _cluster(case):
    return synth.uniform_cluster(case["nodes"], case["gpus"])


def _population(count, jobs, nodes, gpus, seed):
    """Dense int16 candidates, mostly empty rows, made on the GPU in pieces."""
    step = max(1, min(count, (32 * 8192) // jobs))
    out = torch.empty((count, jobs, nodes), dtype=torch.int16, device=GPU)
    for c in range(0, count, step):
        n = min(step, count - c)
        out[c:c + n] = synth.stress_population(n, jobs, nodes, gpus, seed, device=GPU, first_candidate=c)
    return out


def _table(jobs, k_max, n_max, gpus, seed):
    """fp32 [jobs][k_max + 1][n_max + 1] in the shape of the stress workload's tables: K^u, times v
    on several nodes, 1 at (2, 1), 0 where K replicas do not fit N nodes."""
    g = torch.Generator(device=GPU)
    g.manual_seed(seed)
    u = 0.3 + 0.7 * torch.rand(jobs, 1, 1, generator=g, device=GPU)
    v = 0.5 + 0.5 * torch.rand(jobs, 1, 1, generator=g, device=GPU)
    K = torch.arange(k_max + 1, device=GPU, dtype=torch.float32)[None, :, None]
    N = torch.arange(n_max + 1, device=GPU, dtype=torch.float32)[None, None, :]
    val = torch.pow(K.clamp(min=1.0), u) * torch.where(N >= 2, v, torch.ones_like(v)) / torch.pow(torch.full_like(u, 2.0), u)
    return torch.where((N >= 1) & (K >= N) & (K <= N * gpus), val, torch.zeros_like(val)).contiguous()


def prepare(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        st = {"round": _prepare_round, "table": _prepare_table, "generation": _prepare_generation,
              "fitness": _prepare_fitness, "fit": _prepare_fit}[case["kind"]](case, seed, stream)
    st["case"], st["step"] = case, 0
    stream.synchronize()
    return st


def _prepare_round(case, seed, stream):
    cl = _cluster(case)
    jobs = _jobs(case, cl, seed)
    cur = synth.random_feasible_allocation(cl, case["jobs"], seed + 1000, active=jobs.active)
    st = {"sched": _scheduler(case, cl, stream, seed)}
    if case["racks"]:
        a, b = synth.draw_rack_pair(jobs, seed + 2000)
        st["sched"].set_racks(synth.rack_of_nodes(case["nodes"], -(-case["nodes"] // case["racks"])), _dev(a), _dev(b))
    if case["host"]:
        st["jobs"] = api.HostJobs(jobs, torch)
        st["cur"] = torch.from_numpy(cur).pin_memory()
        st["best"] = torch.empty(cur.shape, dtype=torch.int16).pin_memory()
        st["fitness"] = torch.zeros(1, dtype=torch.float32).pin_memory()
    else:
        st["jobs"] = api.DeviceJobs(jobs, GPU, torch)
        st["cur"] = _dev(cur)
        st["best"] = torch.empty(cur.shape, dtype=torch.int16, device=GPU)
        st["fitness"] = torch.zeros(1, dtype=torch.float32, device=GPU)
    return st


def _prepare_table(case, seed, stream):
    cl = _cluster(case)
    jobs = _jobs(case, cl, seed)
    st = {"sched": _scheduler(case, cl, stream, seed), "jobs": api.DeviceJobs(jobs, GPU, torch)}
    if case["samples"]:
        st["samples"] = _dev(synth.make_m_samples(jobs.m0, jobs.m_max_total, case["samples"]))
        st["m_max"] = _dev(jobs.m_max_gpu)
    st["goodput"] = torch.empty(st["sched"].table_shape, dtype=torch.float32, device=GPU)
    st["speedup"] = torch.empty_like(st["goodput"])
    st["argmax"] = torch.empty(st["sched"].table_shape, dtype=torch.int16, device=GPU)     # its 16 bits are unsigned
    return st


def _prepare_generation(case, seed, stream):
    cl = _cluster(case)
    jobs = _jobs(case, cl, seed)
    cur = _dev(synth.random_feasible_allocation(cl, case["jobs"], seed + 1000))
    st = {"sched": _scheduler(case, cl, stream, seed), "jobs": api.DeviceJobs(jobs, GPU, torch), "cur": cur}
    shape = (case["population"], case["jobs"], case["nodes"])
    st["parents"] = torch.empty(shape, dtype=torch.int16, device=GPU)
    st["children"] = torch.empty_like(st["parents"])
    st["sched"].init_population(st["jobs"], cur, st["parents"], round=seed % 1000)
    st["table"] = _table(case["jobs"], cl.k_max, cl.n_max, case["gpus"], seed)
    g = torch.Generator(device=GPU)
    g.manual_seed(seed + 1)
    st["parents_fitness"] = torch.rand(case["population"], generator=g, device=GPU)
    st["fitness"] = torch.empty(case["population"], dtype=torch.float32, device=GPU)
    st["factor"] = torch.empty(case["jobs"], dtype=torch.float32, device=GPU)
    st["sched"].compute_realloc_factor(st["jobs"], st["factor"])
    return st


def _prepare_fitness(case, seed, stream):
    cl = _cluster(case)
    st = {"sched": _scheduler(case, cl, stream, seed)}
    st["pop"] = _population(case["count"], case["jobs"], case["nodes"], case["gpus"], seed)
    st["table"] = _table(case["jobs"], cl.k_max, cl.n_max, case["gpus"], seed)
    st["cur"] = st["factor"] = None
    if case["penalty"]:
        # most candidates of a search keep most rows of the current allocation
        st["cur"] = _population(1, case["jobs"], case["nodes"], case["gpus"], seed + 1)[0].contiguous()
        g = torch.Generator(device=GPU)
        g.manual_seed(seed + 2)
        keep = torch.rand(case["count"], case["jobs"], generator=g, device=GPU) < 0.9
        for c in range(case["count"]):
            st["pop"][c] = torch.where(keep[c][:, None], st["cur"], st["pop"][c])
        st["factor"] = torch.rand(case["jobs"], generator=g, device=GPU)
    if case["racks"]:
        st["sched"].set_racks(synth.rack_of_nodes(case["nodes"], -(-case["nodes"] // case["racks"])))
        N = torch.arange(cl.n_max + 1, device=GPU)
        st["table_rack"] = torch.where(N >= 2, 0.7 * st["table"], torch.zeros_like(st["table"])).contiguous()
    st["fitness"] = torch.empty(case["count"], dtype=torch.float32, device=GPU)
    return st


def _iteration_time(th, K, N, m, s):
    """T_iter of Eq. 11: what a job's profiler would report for (K, N, m, s)."""
    a_g, b_g, a_l, b_l, a_n, b_n, g = th.T
    grad = a_g + b_g * m
    sync = np.where(K < 2, 0.0, np.where(N == 1, a_l + b_l * (K - 2), a_n + b_n * (K - 2)))
    return s * grad + (grad ** g + sync ** g) ** (1.0 / g)


def _prepare_fit(case, seed, stream):
    J, n = case["jobs"], case["observations"]
    jobs = synth.draw_jobs(J, seed, 8, 8, 16)
    offset, K, N, m, s, noise = synth.draw_observations(jobs, n, seed + 1)
    th = np.stack([jobs.alpha_grad, jobs.beta_grad, jobs.alpha_local, jobs.beta_local, jobs.alpha_node, jobs.beta_node,
                   jobs.gamma], axis=1).astype(np.float64)
    T = (_iteration_time(np.repeat(th, n, axis=0), K, N, m, s) * noise).astype(np.float32)
    start = np.tile(np.array([0.1, 0.01, 0.01, 0.01, 0.01, 0.01, 1.0], np.float32), (J, 1))
    st = {"sched": api.Scheduler(node_capacity=np.full(4, 4, np.int16), num_jobs=1, grid_m=1, grid_s=1, population=1,
                                 stream=stream.cuda_stream)}
    st["obs"] = [_dev(a) for a in (offset, K, N, m, s, T, start)]
    st["theta"] = torch.empty((J, 7), dtype=torch.float32, device=GPU)
    st["loss"] = torch.empty(J, dtype=torch.float32, device=GPU)
    return st


# ---- one pass ----------------------------------------------------------------------------------
def run(st):
    case, sched = st["case"], st["sched"]
    kind = case["kind"]
    if kind == "round":
        st["step"] += 1                  # a scheduler numbers its rounds: each draws its own random numbers
        call = sched.schedule_round_host if case["host"] else sched.schedule_round
        call(st["jobs"], st["cur"], st["best"], st["fitness"], round=st["step"], generations=case["generations"])
        return {"best": st["best"], "fitness": st["fitness"]}
    if kind == "table":
        if case["samples"]:
            sched.build_speedup_table_msample(st["jobs"], st["samples"], st["m_max"], st["goodput"], st["speedup"], st["argmax"])
        else:
            sched.build_speedup_table(st["jobs"], st["goodput"], st["speedup"], st["argmax"])
        return {"goodput": st["goodput"], "speedup": st["speedup"], "argmax": st["argmax"]}
    if kind == "generation":
        st["step"] += 1
        sched.ga_generation(st["jobs"], st["parents"], st["parents_fitness"], st["children"], round=1, generation=st["step"])
        sched.eval_fitness(st["children"], st["table"], st["fitness"], p=-1.0, cur=st["cur"], realloc_factor=st["factor"],
                           active=st["jobs"].tensors["active"])
        return {"children": st["children"], "fitness": st["fitness"]}
    if kind == "fitness":
        if case["racks"]:
            sched.eval_fitness_racks(st["pop"], st["table"], st["table_rack"], st["fitness"], p=case["p"], cur=st["cur"],
                                     realloc_factor=st["factor"])
        else:
            sched.eval_fitness(st["pop"], st["table"], st["fitness"], p=case["p"], cur=st["cur"], realloc_factor=st["factor"])
        return {"fitness": st["fitness"]}
    sched.fit_throughput_model(*st["obs"], st["theta"], st["loss"], max_iters=100)
    return {"theta": st["theta"], "loss": st["loss"]}


# ---- what a pass cannot do without ---------------------------------------------------------------
def _pairs(cl):
    """(K, one node or several) pairs that exist on the cluster."""
    fit = np.concatenate([[0], np.cumsum(np.sort(cl.node_capacity.astype(np.int64))[::-1])])
    return sum(int(K <= fit[1]) + int(cl.n_max >= 2 and K >= 2 and K <= fit[min(K, cl.n_max)]) for K in range(1, cl.k_max + 1))


def _table_work(case, cl):
    """Inputs once; per (job, pair, batch size) the two-sided time model with its overlap term, the
    best accumulation count and the comparison: about 40 operations."""
    J = case["jobs"]
    points = case.get("samples", 0) or case["grid_m"]
    return {"bytes": J * (13 * 4 + points * 4), "flops": 40.0 * J * _pairs(cl) * points}


def work(case):
    J = case["jobs"]
    if case["kind"] == "fit":
        # every observation once in, seven parameters out; ten steps, each with the normal equations of
        # 64-bit residuals (about 250 operations an observation) and one trial of the new point (150)
        return {"bytes": J * (case["observations"] * 20 + 7 * 8 + 8), "flops": 10 * 400.0 * J * case["observations"]}
    cl = _cluster(case)
    entries = (cl.k_max + 1) * (cl.n_max + 1)
    mat = J * case["nodes"] * 2
    if case["kind"] == "table":
        w = _table_work(case, cl)
        return {"bytes": w["bytes"] + J * entries * 10, "flops": w["flops"]}
    if case["kind"] == "generation":
        P = case["population"]
        # parents in, children out (the fitness of a child needs nothing that is not in hand while it
        # is made); two draws of the counter-based stream a row, some 80 operations each
        return {"bytes": 2 * P * mat + 8 * P + mat + J * 16 + 4 * J * entries, "flops": 160.0 * P * J}
    if case["kind"] == "fitness":
        # a row's speedup is one table entry
        return {"bytes": case["count"] * (mat + 4 * J + 4) + (mat + 4 * J if case["penalty"] else 0),
                "flops": case["count"] * J * (case["nodes"] * 2.0 + 10)}
    w = _table_work(case, cl)
    P, G = case["population"], case["generations"]
    # job arrays and the current allocation in, the best allocation out; two draws a row and
    # generation, and ten operations to pass the row on
    rows = float(P) * J * case["active"] * (G + 1)
    return {"bytes": w["bytes"] + J * 20 + 2 * mat + 4, "flops": w["flops"] + 170.0 * rows}


def tolerance(case):
    if case["kind"] == "fit":
        # 64-bit steps to a local minimum, rounded to 32 bits: where the error hardly depends on a
        # parameter, that parameter is looser than the rest
        return {"rel": 1e-5, "max": 1e-3}
    if case["kind"] == "table":
        # 32-bit model with approximate exponentials; the best (m, s) of two that tie within it may be either
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-3}
    # matrices are whole numbers and the same for everybody; fitness is a 32-bit mean
    return {"rel": 1e-5, "max": 1e-4}
