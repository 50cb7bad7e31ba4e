"""Rounds about the lines where the one-launch search changes its blocks: how many candidates share an SM and how many
jobs keep their records in shared memory.  (Which blocks a round got is not looked at.)  Bit for bit the dense entry points one by
one."""
import pytest
import torch

import test_gpu_round_shapes as shapes

pytestmark = pytest.mark.gpu

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148

# as in test_gpu_round_shapes: nodes, GPUs per node, jobs, population, generations, nodes per rack, active, perturbation
KINDS = [
    # a block or several an SM, records in shared memory or not
    (20, 4, 256, SMS, 4, 0, 1.0, 0.2), (20, 4, 256, SMS + 1, 4, 6, 1.0, 0.2), (20, 4, 257, SMS, 4, 6, 1.0, 0.2),
    (20, 4, 257, SMS + 1, 4, 0, 1.0, 0.2), (12, 8, 1024, 30, 3, 4, 0.8, 0.1), (12, 8, 1025, 30, 3, 0, 1.0, 0.1),
    (3, 8, 2720, 20, 3, 0, 1.0, 0.1), (3, 8, 2810, 20, 3, 2, 0.9, 0.1), (12, 8, 1204, 2 * SMS, 2, 0, 1.0, 0.1),
    (12, 8, 1206, 2 * SMS, 2, 0, 1.0, 0.1), (12, 8, 1206, 2 * SMS + 1, 2, 0, 1.0, 0.1), (6, 4, 8192, 7, 2, 0, 1.0, 0.1),
    (12, 8, 700, 2 * SMS, 3, 0, 1.0, 0.1), (12, 8, 300, 2 * SMS + 1, 3, 0, 1.0, 0.1), (20, 4, 64, 2 * SMS, 4, 0, 1.0, 0.2),
    (20, 4, 64, 2 * SMS + 1, 4, 0, 0.5, 0.2), (20, 4, 64, 3 * SMS + 1, 4, 5, 1.0, 0.2), (64, 4, 900, 200, 3, 0, 1.0, 0.9),
    # a thread per changed row: more perturbed rows than draws are kept of, racks, wide rows
    (64, 2, 900, 2 * SMS + 1, 3, 16, 0.8, 0.9), (30, 4, 600, 2 * SMS + 1, 3, 0, 1.0, 0.14),
    # smaller blocks, and more candidates than blocks
    (20, 4, 30, 4 * SMS, 4, 0, 1.0, 0.2), (20, 4, 30, 4 * SMS + 1, 4, 6, 1.0, 0.2), (20, 4, 30, 5 * SMS + 1, 4, 0, 0.7, 0.2),
    (20, 4, 30, 6 * SMS + 1, 4, 6, 1.0, 0.9), (20, 4, 30, 8 * SMS, 4, 0, 1.0, 0.2), (20, 4, 30, 8 * SMS + 1, 4, 6, 1.0, 0.2),
    (20, 4, 250, 8 * SMS, 3, 0, 1.0, 0.2), (1, 4, 1, 3, 3, 0, 1.0, 1.0),
    # enough generations for the terms to be copied, and one fewer
    (6, 4, 41, 20, 100, 2, 1.0, 0.1), (6, 4, 41, 20, 101, 2, 0.9, 0.1), (6, 4, 41, SMS + 5, 101, 0, 1.0, 0.1),
    (6, 4, 40, 20, 39, 0, 1.0, 0.1), (6, 4, 40, SMS + 5, 40, 2, 0.9, 0.1),
    (2, 4, 300, 12, 101, 0, 1.0, 0.1), (3, 2, 280, 2 * SMS, 101, 2, 1.0, 0.1),
]


@pytest.mark.parametrize("shape", KINDS, ids=lambda s: "-".join(str(x) for x in s))
@pytest.mark.parametrize("start", ["none", "feasible", "raw"])
def test_rounds_at_the_kinds_edges(shape, start):
    shapes.test_round_equals_stepwise("flow", shape, start)


# nodes with more occupants than a group of lanes takes, in every kind of block: within the lists, beyond them (many GPUs a
# node and rows everywhere), with racks, inactive jobs and rows of more nodes than a record holds
CROWDS = [
    (3, 8, 200, 40, 5, 0, 1.0, 0.5), (4, 4, 900, 30, 4, 2, 0.8, 0.3), (4, 4, 300, 200, 3, 0, 1.0, 0.3), (4, 8, 1100, 160, 3, 0, 1.0, 0.2),
    (2, 300, 1300, 20, 3, 0, 1.0, 0.3), (2, 300, 250, 200, 3, 1, 1.0, 0.3), (20, 2, 250, 100, 12, 5, 1.0, 0.9), (20, 2, 250, 460, 6, 0, 1.0, 0.9),
]


@pytest.mark.parametrize("shape", CROWDS, ids=lambda s: "-".join(str(x) for x in s))
@pytest.mark.parametrize("start", ["none", "feasible", "raw"])
def test_rounds_with_crowded_nodes(shape, start):
    shapes.test_round_equals_stepwise("flow", shape, start)


# candidates, elite children, share of rows perturbed at first and per generation: ranks of few keys above the bound, of
# more (ties in a converged population), of as many as there are, and ranks beyond a warp's lanes
@pytest.mark.parametrize("P,elite,init,mutate", [(64, 4, 0.0, 0.0), (65, 31, 0.0, 0.0), (300, 16, 0.01, 0.0), (300, 31, 0.01, 0.01),
                                                 (300, 32, 0.3, 0.05), (148, 148, 0.3, 0.0), (500, 200, 0.05, 0.01)])
def test_elite_candidates_of_a_round(P, elite, init, mutate):
    import numpy as np
    from helpers import with_fair_share
    from paper_2008_12260_b200 import api, synth

    cfg = synth.Config("ranks", 12, 4, 30, 3, 16, 8, P, 6, num_elite=elite, mutate_prob=mutate, init_prob=init, with_history=True)
    cl = cfg.cluster()
    jobs = with_fair_share(cfg.jobs(), cl)
    s = api.scheduler_for(cfg, stream=torch.cuda.current_stream().cuda_stream)
    dj = api.DeviceJobs(jobs, "cuda", torch)
    cur = torch.from_numpy(synth.random_feasible_allocation(cl, cfg.num_jobs, 5)).cuda()
    best, bf = torch.empty((cfg.num_jobs, 12), dtype=torch.int16, device="cuda"), torch.zeros(1, device="cuda")
    pop, fit = torch.empty((P, cfg.num_jobs, 12), dtype=torch.int16, device="cuda"), torch.empty(P, device="cuda")
    sp, rf = torch.empty(s.table_shape, device="cuda"), torch.empty(cfg.num_jobs, device="cuda")
    s.schedule_round(dj, cur, best, bf, round=2, generations=6)
    s.get_population(pop, fit)
    s.build_speedup_table(dj, None, sp, None)
    s.compute_realloc_factor(dj, rf)
    a, b, f = torch.empty_like(pop), torch.empty_like(pop), torch.empty_like(fit)
    s.init_population(dj, cur, a, round=2)
    for g in range(7):
        s.eval_fitness(a, sp, f, p=cfg.p, cur=cur, realloc_factor=rf, active=dj.tensors["active"])
        if g < 6:                 # the rank of a child's parent is checked against a plain sort as well
            order = np.argsort(-f.cpu().numpy(), kind="stable")
            s.ga_generation(dj, a, f, b, round=2, generation=g)
            for c in range(0, elite, 7):
                assert torch.equal(b[c], a[int(order[c])])
            a, b = b, a
    s.sync_status()
    assert torch.equal(a, pop) and torch.equal(f.view(torch.int32), fit.view(torch.int32))
    s.close()
