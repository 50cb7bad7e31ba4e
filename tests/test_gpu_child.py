"""Dense operators with a block (or a cluster of blocks) per child: rows of every width relative to a 16-byte vector,
buffers that begin between two vectors, crowded nodes (more occupants than a list holds), entries out of range,
full rows (every vector of a tile queued), children split over several blocks.  Bit-exact against the oracle,
whose code knows none of these cases."""
import numpy as np
import pytest

from paper_2008_12260_b200 import synth

pytestmark = pytest.mark.gpu


class _Jobs:
    def __init__(self, k_cap, active):
        self.k_cap, self.active = k_cap, active


def _unaligned(torch, a, shift):
    """A device copy of `a` that begins `shift` entries behind a 16-byte boundary, with guards around it."""
    flat = torch.full((a.size + 32,), 77, dtype=torch.int16, device="cuda:0")
    view = flat[8 + shift:8 + shift + a.size].view(a.shape)
    view.copy_(torch.from_numpy(a))
    return flat, view


def _guards_ok(flat, shift, size):
    return bool((flat[:8 + shift] == 77).all()) and bool((flat[8 + shift + size:] == 77).all())


# nodes, jobs, population, density of the raw matrices, shifts of parents and children
CASES = [
    (1, 3, 5, 0.9, 1, 0), (7, 33, 9, 0.3, 0, 3), (8, 33, 9, 0.3, 0, 0), (8, 33, 9, 0.3, 4, 0), (9, 1, 4, 0.5, 7, 2),
    (31, 40, 7, 0.2, 0, 0), (33, 257, 200, 0.05, 5, 6), (75, 300, 3, 0.1, 0, 0), (255, 70, 5, 0.02, 1, 7),
    (256, 130, 4, 0.02, 0, 0), (256, 64, 4, 1.0, 0, 5), (257, 65, 3, 0.02, 0, 0), (448, 40, 3, 0.05, 3, 3), (504, 33, 3, 0.05, 0, 0),
    (511, 37, 3, 0.05, 0, 1), (512, 37, 3, 1.0, 0, 0), (512, 37, 3, 0.3, 0, 0), (512, 37, 3, 0.3, 2, 0), (16, 1000, 2, 0.2, 0, 0),
]


@pytest.mark.parametrize("nodes,J,P,density,shift_in,shift_out", CASES)
def test_children_of_any_width(oracle, nodes, J, P, density, shift_in, shift_out):
    import torch
    from paper_2008_12260_b200 import api

    rng = np.random.default_rng(nodes * 1000 + J)
    cl = synth.Cluster(rng.integers(0, 9, nodes).astype(np.int16)) if nodes > 1 else synth.uniform_cluster(1, 4)
    if int(np.maximum(cl.node_capacity, 0).sum()) == 0:
        cl = synth.uniform_cluster(nodes, 4)
    raw = synth.random_raw_population(P, J, cl, seed=nodes + J, density=density, v_hi=9)
    raw[-1, 0, -1], raw[0, 0, 0] = 30000, -5                # out of range, at both ends of the buffer
    k_cap = rng.integers(0, cl.k_max + 3, J).astype(np.int32)
    active = (rng.uniform(size=J) < 0.85).astype(np.uint8)
    fit = rng.uniform(0.1, 1.0, P).astype(np.float32)
    thr, elite, seed = synth.prob_to_threshold(0.3), min(2, P - 1), 77
    s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=J, grid_m=1, grid_s=1, population=P, thr_mutate=thr,
                      thr_init=thr, num_elite=elite, seed=seed, stream=torch.cuda.current_stream().cuda_stream)
    dj = api.DeviceJobs(_Jobs(k_cap, active), "cuda:0", torch)
    _, parents = _unaligned(torch, raw, shift_in)
    out_flat, out = _unaligned(torch, np.full(raw.shape, 5, np.int16), shift_out)

    s.ga_generation(dj, parents, torch.from_numpy(fit).cuda(), out, round=2, generation=3)
    ref = oracle.ga_generation(raw, fit, cl.node_capacity, k_cap, cl.k_max, cl.n_max, elite, thr, seed, 2, 3, active=active)
    assert np.array_equal(out.cpu().numpy(), ref)

    s.init_population(dj, parents[0], out, round=4)
    ref = oracle.init_population(P, raw[0], J, cl.node_capacity, k_cap, cl.k_max, cl.n_max, thr, seed, 4, active=active)
    assert np.array_equal(out.cpu().numpy(), ref)

    out.copy_(torch.from_numpy(raw))
    s.repair_population(dj, out, round=5, generation=6, first_candidate=9)
    got = out.cpu().numpy()
    for c in range(P):
        ref = oracle.repair(raw[c], cl.node_capacity, k_cap, cl.k_max, cl.n_max, seed, 5, 9 + c, 6, active=active)
        assert np.array_equal(got[c], ref), c
    assert _guards_ok(out_flat, shift_out, raw.size)
    s.sync_status()
    s.close()


# population, elite children: as many as lanes, more, everybody; keys in one turn of a block and in many
@pytest.mark.parametrize("P,elite", [(1, 1), (33, 33), (256, 40), (257, 256), (5121, 70), (7361, 33)])
@pytest.mark.parametrize("values", [0, 5, 1])           # different fitness values (0: all of them differ)
@pytest.mark.parametrize("nodes", [3, 8])
def test_elite_children_of_any_rank(oracle, P, elite, values, nodes):
    import torch
    from paper_2008_12260_b200 import api

    rng = np.random.default_rng(P + elite + values)
    cl = synth.uniform_cluster(nodes, 4)
    J, thr, seed = 2, synth.prob_to_threshold(0.3), 5
    raw = synth.random_raw_population(P, J, cl, seed=P, density=0.4, v_hi=4)
    fit = (rng.integers(0, values, P) - 2).astype(np.float32) if values else rng.permutation(P).astype(np.float32)
    k_cap, active = np.full(J, cl.k_max, np.int32), np.ones(J, np.uint8)
    s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=J, grid_m=1, grid_s=1, population=P, thr_mutate=thr,
                      num_elite=elite, seed=seed, stream=torch.cuda.current_stream().cuda_stream)
    out = torch.empty(raw.shape, dtype=torch.int16, device="cuda:0")
    s.ga_generation(api.DeviceJobs(_Jobs(k_cap, active), "cuda:0", torch), torch.from_numpy(raw).cuda(),
                    torch.from_numpy(fit).cuda(), out, round=1, generation=2)
    ref = oracle.ga_generation(raw, fit, cl.node_capacity, k_cap, cl.k_max, cl.n_max, elite, thr, seed, 1, 2, active=active)
    assert np.array_equal(out.cpu().numpy(), ref)
    s.sync_status()
    s.close()


# nodes, GPUs a node, jobs, children, density: about as many occupants a node as a group of lanes takes (16), as the blocks' lists
# hold (16 to 768, by the node's size and the rows perturbed), and more; one block and several; nodes larger than what lies on
# them, and one without any GPUs
CROWDS = [(1, 3, 17, 3, 1.0), (1, 3, 26, 3, 1.0), (1, 500, 600, 3, 1.0), (1, 500, 680, 3, 1.0), (1, 2047, 700, 1, 1.0), (1, 2047, 1280, 2, 1.0),
          (3, 8, 2000, 1, 0.3), (3, 8, 2000, 1, 0.45), (8, 0, 200, 4, 0.09), (8, 40, 1024, 2, 0.06), (8, 40, 1024, 2, 0.6),
          (9, 8, 3000, 300, 0.029), (64, 8, 700, 3, 0.028), (64, 8, 4000, 2, 0.007), (250, 4, 300, 3, 0.06), (256, 4, 300, 3, 0.06),
          (512, 4, 120, 2, 0.14)]


@pytest.mark.parametrize("nodes,gpus,J,P,density", CROWDS)
def test_crowded_nodes(oracle, nodes, gpus, J, P, density):
    import torch
    from paper_2008_12260_b200 import api

    rng = np.random.default_rng(nodes + J)
    cap = np.full(nodes, max(gpus, 1), np.int16)
    cap[nodes // 2] = gpus                                  # (0: a node without any)
    raw = synth.random_raw_population(P, J, synth.Cluster(cap), seed=nodes + J, density=density, v_hi=4)
    raw[:, :, 0] = rng.integers(0, 3, (P, J))
    k_max, n_max = 64, min(nodes, 64)
    k_cap, active = rng.integers(1, 40, J).astype(np.int32), (rng.uniform(size=J) < 0.9).astype(np.uint8)
    fit, thr, seed = rng.uniform(0.1, 1.0, P).astype(np.float32), synth.prob_to_threshold(0.2), 9
    s = api.Scheduler(node_capacity=cap, num_jobs=J, grid_m=1, grid_s=1, population=P, thr_mutate=thr, thr_init=thr, num_elite=0,
                      seed=seed, k_max=k_max, n_max=n_max, stream=torch.cuda.current_stream().cuda_stream)
    dj = api.DeviceJobs(_Jobs(k_cap, active), "cuda:0", torch)
    parents, out = torch.from_numpy(raw).cuda(), torch.empty(raw.shape, dtype=torch.int16, device="cuda:0")
    s.ga_generation(dj, parents, torch.from_numpy(fit).cuda(), out, round=2, generation=3)
    ref = oracle.ga_generation(raw, fit, cap, k_cap, k_max, n_max, 0, thr, seed, 2, 3, active=active)
    assert np.array_equal(out.cpu().numpy(), ref)
    s.repair_population(dj, parents, round=5, generation=6, first_candidate=9)
    got = parents.cpu().numpy()
    for c in range(0, P, max(1, P // 4)):
        assert np.array_equal(got[c], oracle.repair(raw[c], cap, k_cap, k_max, n_max, seed, 5, 9 + c, 6, active=active)), c
    s.sync_status()
    s.close()


# beyond 65535 jobs a node's counters no longer do: rows of whole vectors on the batched kernels, others a row and a column at a time
@pytest.mark.parametrize("nodes,shift", [(8, 0), (8, 1), (9, 0), (24, 0)])
def test_more_jobs_than_a_nodes_counters_hold(oracle, nodes, shift):
    import torch
    from paper_2008_12260_b200 import api

    J, P, thr, seed = 65541, 3, synth.prob_to_threshold(0.2), 4
    rng = np.random.default_rng(nodes)
    cl = synth.uniform_cluster(nodes, 8)
    raw = synth.random_raw_population(P, J, cl, seed=nodes, density=0.0005, v_hi=9)
    raw[1, :40, 2] = 3                                      # more occupants of a batch of rows than are listed
    k_cap, active = rng.integers(0, cl.k_max + 3, J).astype(np.int32), (rng.uniform(size=J) < 0.9).astype(np.uint8)
    fit = rng.uniform(0.1, 1.0, P).astype(np.float32)
    s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=J, grid_m=1, grid_s=1, population=P, thr_mutate=thr, thr_init=thr,
                      num_elite=1, seed=seed, stream=torch.cuda.current_stream().cuda_stream)
    dj = api.DeviceJobs(_Jobs(k_cap, active), "cuda:0", torch)
    _, parents = _unaligned(torch, raw, shift)
    out_flat, out = _unaligned(torch, np.full(raw.shape, 5, np.int16), shift)
    s.set_kernel_timing(True)
    s.ga_generation(dj, parents, torch.from_numpy(fit).cuda(), out, round=2, generation=3)
    ran = {name for name, (ms, n) in s.read_kernel_timing().items() if n}
    assert "cols" in ran and ("rank" in ran) == (nodes % 8 != 0 or shift != 0)
    ref = oracle.ga_generation(raw, fit, cl.node_capacity, k_cap, cl.k_max, cl.n_max, 1, thr, seed, 2, 3, active=active)
    assert np.array_equal(out.cpu().numpy(), ref)
    s.init_population(dj, parents[1], out, round=4)
    ref = oracle.init_population(P, raw[1], J, cl.node_capacity, k_cap, cl.k_max, cl.n_max, thr, seed, 4, active=active)
    assert np.array_equal(out.cpu().numpy(), ref)
    s.repair_population(dj, parents, round=5, generation=6, first_candidate=9)
    got = parents.cpu().numpy()
    for c in range(P):
        assert np.array_equal(got[c], oracle.repair(raw[c], cl.node_capacity, k_cap, cl.k_max, cl.n_max, seed, 5, 9 + c, 6, active=active)), c
    assert _guards_ok(out_flat, shift, raw.size)
    s.sync_status()
    s.close()


# nodes, jobs, children, share of rows perturbed, what the three operators run on: so few children of so many rows that a block per
# 256 rows is quicker ("cols": with the work-list repair behind it), the same with crowded nodes, and either side of that
MANY_ROWS = [(256, 4096, 1, 0.02, "cols cols cols"), (64, 17000, 3, 0.01, "cols cols cols"), (512, 1900, 65, 0.01, "cols cols cols"),
             (16, 8193, 4, 0.01, "cols cols rows"), (16, 17000, 2, 0.3, "rows rows rows"), (256, 1024, 2, 0.02, "rows rows rows"),
             (512, 1000, 65, 0.01, "rows rows rows")]


@pytest.mark.parametrize("nodes,J,P,share,routes", MANY_ROWS)
def test_few_children_of_many_rows(oracle, nodes, J, P, share, routes):
    _three_operators(oracle, nodes, J, P, share, routes.split())


def test_few_children_of_many_rows_without_scratch(oracle):
    """A captured call whose scratch is not there yet: one launch a child instead."""
    import torch
    from paper_2008_12260_b200 import api

    nodes, J, P, seed = 256, 4096, 2, 3
    cl = synth.uniform_cluster(nodes, 4)
    raw = synth.random_raw_population(P, J, cl, seed=1, density=0.002, v_hi=6)
    k_cap, active = np.full(J, cl.k_max, np.int32), np.ones(J, np.uint8)
    stream = torch.cuda.Stream()
    s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=J, grid_m=1, grid_s=1, population=P, thr_mutate=1 << 26, seed=seed,
                      stream=stream.cuda_stream)
    dj = api.DeviceJobs(_Jobs(k_cap, active), "cuda:0", torch)
    _, aside = _unaligned(torch, raw, 1)
    pop = torch.from_numpy(raw).cuda()
    torch.cuda.synchronize()
    s.repair_population(dj, aside, round=5, generation=6)   # (rows between two vectors: no scratch)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        s.repair_population(dj, pop, round=5, generation=6)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(pop, aside)
    got = pop.cpu().numpy()
    for c in range(P):
        assert np.array_equal(got[c], oracle.repair(raw[c], cl.node_capacity, k_cap, cl.k_max, cl.n_max, seed, 5, c, 6, active=active)), c
    s.sync_status()
    s.set_kernel_timing(True)
    s.repair_population(dj, pop, round=5, generation=6)
    assert s.read_kernel_timing()["cols"][1] == 1
    s.close()


# many children of a few rows: a warp a row and a thread a node, unless ranks are wanted
@pytest.mark.parametrize("nodes,J,P,routes", [(3, 1, 1100, "cols rows cols"), (20, 24, 1100, "cols rows cols"), (301, 16, 1100, "cols rows cols"),
                                              (301, 17, 1100, "rows rows rows"), (20, 25, 1100, "rows rows rows"),
                                              (8, 4, 1100, "rows rows rows"), (20, 4, 500, "rows rows rows")])
def test_many_children_of_few_rows(oracle, nodes, J, P, routes):
    _three_operators(oracle, nodes, J, P, 0.2, routes.split())


def _three_operators(oracle, nodes, J, P, share, routes):
    """Initial population, generation and repair, the kernels they run on ("rows": child_kernel alone) and their results."""
    import torch
    from paper_2008_12260_b200 import api

    thr, seed, elite = synth.prob_to_threshold(share), 11, 1 if P > 1 else 0
    rng = np.random.default_rng(nodes + J)
    cl = synth.uniform_cluster(nodes, 4)
    raw = synth.random_raw_population(P, J, cl, seed=nodes + P, density=0.002 if J > 100 else 0.1, v_hi=6)
    k_cap, active = rng.integers(0, cl.k_max + 3, J).astype(np.int32), (rng.uniform(size=J) < 0.9).astype(np.uint8)
    fit = rng.uniform(0.1, 1.0, P).astype(np.float32)
    s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=J, grid_m=1, grid_s=1, population=P, thr_mutate=thr, thr_init=thr,
                      num_elite=elite, seed=seed, stream=torch.cuda.current_stream().cuda_stream)
    dj = api.DeviceJobs(_Jobs(k_cap, active), "cuda:0", torch)
    parents, out = torch.from_numpy(raw).cuda(), torch.empty(raw.shape, dtype=torch.int16, device="cuda:0")
    s.set_kernel_timing(True)
    ran = lambda: "cols" if s.read_kernel_timing()["cols"][1] else "rows"
    some = sorted({0, 1 % P, P // 2, P - 1})                # (the oracle takes its time over large populations)

    s.init_population(dj, parents[0], out, round=4)
    used = [ran()]
    got = out.cpu().numpy()
    want = oracle.init_population(P, raw[0], J, cl.node_capacity, k_cap, cl.k_max, cl.n_max, thr, seed, 4, active=active)
    assert np.array_equal(got, want)
    s.ga_generation(dj, parents, torch.from_numpy(fit).cuda(), out, round=2, generation=3)
    used.append(ran())
    want = oracle.ga_generation(raw, fit, cl.node_capacity, k_cap, cl.k_max, cl.n_max, elite, thr, seed, 2, 3, active=active)
    assert np.array_equal(out.cpu().numpy(), want)
    s.repair_population(dj, parents, round=5, generation=6, first_candidate=9)
    used.append(ran())
    got = parents.cpu().numpy()
    for c in some:
        assert np.array_equal(got[c], oracle.repair(raw[c], cl.node_capacity, k_cap, cl.k_max, cl.n_max, seed, 5, 9 + c, 6, active=active)), c
    assert used == routes
    s.sync_status()
    s.close()
