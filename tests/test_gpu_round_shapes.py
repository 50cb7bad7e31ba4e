"""Rounds at the shapes where their kernels change: node counts that are no multiple of a row's
pieces, racks, few and many jobs, inactive jobs, populations larger than the GPU holds blocks, elites; in one
launch, where a budget can ask for it on the row store, and without any budget on dense matrices.  A round must equal, bit for bit, the same round
made of the dense entry points called one by one (which other tests pin to the oracle)."""
import numpy as np
import pytest

from helpers import check_route, feasible, store_budget, with_fair_share
from paper_2008_12260_b200 import synth

pytestmark = pytest.mark.gpu

# nodes, GPUs per node, jobs, population, generations, nodes per rack (0: none), share of active jobs, perturbation
SHAPES = [
    (1, 8, 5, 4, 3, 0, 1.0, 0.5), (3, 4, 9, 33, 6, 2, 1.0, 0.3), (7, 8, 41, 100, 8, 0, 0.5, 0.1),
    (33, 4, 64, 20, 8, 8, 1.0, 0.2), (75, 8, 210, 40, 6, 0, 1.0, 0.1), (75, 2, 300, 20, 6, 20, 0.7, 0.9),
    (129, 4, 257, 16, 5, 0, 1.0, 0.3), (505, 2, 270, 9, 4, 100, 1.0, 0.4), (512, 4, 33, 12, 5, 64, 1.0, 1.0),
    (40, 2, 6, 24, 40, 10, 1.0, 0.9), (16, 4, 256, 64, 6, 0, 0.3, 0.2), (32, 4, 96, 100, 12, 8, 1.0, 0.08),
    (13, 96, 300, 24, 6, 0, 1.0, 0.3), (9, 200, 50, 24, 6, 4, 1.0, 0.5),
    # more candidates than blocks fit the GPU at once; one candidate; more elites than a warp has lanes
    (16, 4, 270, 700, 3, 0, 1.0, 0.05), (8, 4, 40, 2500, 3, 0, 1.0, 0.1), (8, 4, 20, 1, 5, 0, 1.0, 0.5),
    (24, 4, 70, 90, 6, 6, 0.6, 0.2),
]


@pytest.mark.parametrize("route,shape", [("flow", s) for s in SHAPES] + [("store", s) for s in SHAPES if s[2] > 48] +
                         [("dense", s) for s in SHAPES],
                         ids=lambda s: s if isinstance(s, str) else "-".join(str(x) for x in s))
@pytest.mark.parametrize("start", ["none", "feasible", "raw"])
def test_round_equals_stepwise(route, shape, start):
    import torch
    from paper_2008_12260_b200 import api

    NN, gpn, J, P, gens, per_rack, active, mutate = shape
    cfg = synth.Config("shape", NN, gpn, J, NN + J, 16, 8, P, gens, num_elite=min(P, 40 if P == 90 else J % 3), mutate_prob=mutate, init_prob=0.3,
                       with_history=True, p=-1.0 if J % 2 else 0.5)
    cl = cfg.cluster()
    jobs = cfg.jobs()
    rng = np.random.default_rng(J)
    if active < 1.0:
        jobs.active = (rng.random(J) < active).astype(np.uint8)
        jobs.active[J // 2] = 1
    jobs.k_cap[::5] = rng.integers(0, 5, jobs.k_cap[::5].shape[0])
    jobs = with_fair_share(jobs, cl)
    cur = None
    if start == "feasible":
        cur = synth.random_feasible_allocation(cl, J, 5, active=jobs.active)
    elif start == "raw":
        cur = synth.random_raw_population(1, J, cl, 6, density=0.3, v_hi=2 * gpn)[0]
    dev = "cuda"
    s = api.scheduler_for(cfg, stream=torch.cuda.current_stream().cuda_stream)
    if route != "flow":
        s.set_store_budget(store_budget(cfg) if route == "store" else 0)
    s.set_kernel_timing(True)
    dj = api.DeviceJobs(jobs, dev, torch)
    ar, br = (torch.from_numpy(x).cuda() for x in synth.draw_rack_pair(jobs, 9))
    if per_rack:
        s.set_racks(synth.rack_of_nodes(NN, per_rack), ar, br)
    d_cur = None if cur is None else torch.from_numpy(cur).cuda()
    best = torch.full((J, NN), -1, dtype=torch.int16, device=dev)
    bf = torch.zeros(1, dtype=torch.float32, device=dev)
    pop = torch.empty((P, J, NN), dtype=torch.int16, device=dev)
    fit = torch.empty(P, dtype=torch.float32, device=dev)
    s.schedule_round(dj, d_cur, best, bf, round=2, generations=gens)
    s.sync_status()
    check_route(s, route, summaries=NN % 8 == 0 and not per_rack)
    s.set_kernel_timing(False)
    s.get_population(pop, fit)

    sp = torch.empty(s.table_shape, dtype=torch.float32, device=dev)
    spr = torch.empty_like(sp)
    s.build_speedup_table(dj, None, sp, None)
    if per_rack:
        s.build_speedup_table_rack(dj, ar, br, None, spr, None)
    kw = dict(p=cfg.p, active=dj.tensors["active"])
    if cur is not None:
        rf = torch.empty(J, dtype=torch.float32, device=dev)
        s.compute_realloc_factor(dj, rf)
        kw.update(cur=d_cur, realloc_factor=rf)

    def evaluate(x, out):
        if per_rack:
            s.eval_fitness_racks(x, sp, spr, out, **kw)
        else:
            s.eval_fitness(x, sp, out, **kw)

    a, b, f = torch.empty_like(pop), torch.empty_like(pop), torch.empty_like(fit)
    s.init_population(dj, d_cur, a, round=2)
    evaluate(a, f)
    for g in range(gens):
        s.ga_generation(dj, a, f, b, round=2, generation=g)
        a, b = b, a
        evaluate(a, f)
    s.sync_status()
    assert torch.equal(a, pop)
    assert torch.equal(f.view(torch.int32), fit.view(torch.int32))
    i = int(torch.argmax(fit))
    assert torch.equal(best, pop[i]) and bf.item() == fit[i].item()
    k_cap = np.minimum(np.maximum(jobs.k_cap, 0), cl.k_max)
    for c in range(0, P, 3):
        assert feasible(pop[c].cpu().numpy(), cl.node_capacity, k_cap, cl.n_max)
    s.close()


@pytest.mark.parametrize("shape", [(16, 4, 48, 148, 60), (75, 8, 300, 700, 12), (8, 4, 20, 2500, 20)],
                         ids=lambda s: "-".join(str(x) for x in s))
def test_rows_handed_from_block_to_block_arrive(shape):
    """Blocks read rows that other blocks have just published, for many generations and many times over:
    every repetition must be the same round, bit for bit, and the first the dense entry points'."""
    import torch
    from paper_2008_12260_b200 import api

    NN, gpn, J, P, gens = shape
    cfg = synth.Config("hand-over", NN, gpn, J, 3, 16, 8, P, gens, num_elite=4, mutate_prob=0.3, init_prob=0.5,
                       with_history=True)
    cl = cfg.cluster()
    jobs = with_fair_share(cfg.jobs(), cl)
    cur = synth.random_feasible_allocation(cl, J, 5, active=jobs.active)
    st = torch.cuda.Stream()
    s = api.scheduler_for(cfg, stream=st.cuda_stream)
    with torch.cuda.stream(st):
        dj = api.DeviceJobs(jobs, "cuda", torch)
        d_cur = torch.from_numpy(cur).cuda()
        best, bf = torch.empty((J, NN), dtype=torch.int16, device="cuda"), torch.zeros(1, device="cuda")
        pop, fit = torch.empty((P, J, NN), dtype=torch.int16, device="cuda"), torch.empty(P, device="cuda")
        sp, rf = torch.empty(s.table_shape, device="cuda"), torch.empty(J, device="cuda")
        s.build_speedup_table(dj, None, sp, None)
        s.compute_realloc_factor(dj, rf)
        a, b, f = torch.empty_like(pop), torch.empty_like(pop), torch.empty_like(fit)
        kw = dict(p=cfg.p, cur=d_cur, realloc_factor=rf, active=dj.tensors["active"])
        s.init_population(dj, d_cur, a, round=1)
        s.eval_fitness(a, sp, f, **kw)
        for g in range(gens):
            s.ga_generation(dj, a, f, b, round=1, generation=g)
            a, b = b, a
            s.eval_fitness(a, sp, f, **kw)
        for k in range(20):
            s.schedule_round(dj, d_cur, best, bf, round=1 + k % 2, generations=gens)
            if k % 2:
                continue
            s.get_population(pop, fit)
            s.sync_status()
            assert torch.equal(pop, a) and torch.equal(fit.view(torch.int32), f.view(torch.int32)), k
    s.close()
