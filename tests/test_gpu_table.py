"""Parity of build_speedup_table (CUDA, fp32) against the fp64 oracle."""
import numpy as np
import pytest

from helpers import assert_close, check_table, setup, with_fair_share
from paper_2008_12260_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    from paper_2008_12260_b200 import api
    assert torch.cuda.is_available()
    return torch, api


def _gpu_table(gpu, cl, jobs, grid_s, k_max=None, n_max=None, want_goodput=True, want_argmax=True):
    torch, api = gpu
    dev = torch.device("cuda:0")
    s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=jobs.num_jobs, grid_m=jobs.m_grid.shape[1],
                      grid_s=grid_s, population=1, k_max=k_max, n_max=n_max,
                      stream=torch.cuda.current_stream().cuda_stream)
    dj = api.DeviceJobs(jobs, dev, torch)
    gp = torch.full(s.table_shape, -1.0, dtype=torch.float32, device=dev) if want_goodput else None
    sp = torch.full(s.table_shape, -1.0, dtype=torch.float32, device=dev)
    am = torch.full(s.table_shape, 7, dtype=torch.uint16, device=dev) if want_argmax else None
    s.build_speedup_table(dj, gp, sp, am)
    s.sync_status()
    out = (None if gp is None else gp.cpu().numpy(), sp.cpu().numpy(),
           None if am is None else am.cpu().numpy())
    s.close()
    return out


@pytest.mark.parametrize("cfg", [synth.TINY, synth.TESTBED], ids=lambda c: c.name)
def test_table_matches_oracle(gpu, oracle, cfg):
    cl, jobs = setup(cfg)
    gp, sp, am = _gpu_table(gpu, cl, jobs, cfg.grid_s)
    gp_r, sp_r, am_r = oracle.build_speedup_table(jobs, cl.node_capacity, cl.k_max, cl.n_max, cfg.grid_s)
    ndiff = check_table(oracle, jobs, cfg.grid_s, gp, sp, am, gp_r, sp_r, am_r)
    assert ndiff < 0.05 * am.size
    fk, fn = int(jobs.fair_k[0]), int(jobs.fair_n[0])
    assert np.all(sp[:, fk, fn] == 1.0)       # Eq. 15: exactly one at the fair share


def test_large_config_sampled_jobs(gpu, oracle):
    """Full-size launch (1024 jobs, 128 x 32 grid); the oracle checks a sample of jobs."""
    cfg = synth.LARGE
    cl, jobs = setup(cfg)
    gp, sp, am = _gpu_table(gpu, cl, jobs, cfg.grid_s)
    idx = np.unique(np.concatenate([np.arange(0, 1024, 16), [1, 17, 255, 256, 511, 777, 1000, 1023]]))   # 71 jobs
    sub = jobs.take(idx)
    gp_r, sp_r, am_r = oracle.build_speedup_table(sub, cl.node_capacity, cl.k_max, cl.n_max, cfg.grid_s)
    check_table(oracle, sub, cfg.grid_s, gp[idx], sp[idx], am[idx], gp_r, sp_r, am_r)
    # properties that hold for every job at any size
    assert np.all(sp[:, int(jobs.fair_k[0]), int(jobs.fair_n[0])] == 1.0)
    assert np.all(gp[:, 0, :] == 0) and np.all(gp[:, :, 0] == 0)
    K = np.arange(65)[:, None]; N = np.arange(65)[None, :]
    valid = (N >= 1) & (K >= N) & (K <= 8 * N)
    assert np.all((gp > 0) == valid[None])
    assert np.all(gp[:, 2:9, 1] >= gp[:, 2:9, 2])           # local sync never slower than node sync here
    for K_ in (16, 33, 64):                                 # Eq. 9: N >= 2 columns agree
        cols = [n for n in range(2, 65) if valid[K_, n]]
        assert np.all(gp[:, K_, cols] == gp[:, K_, cols[:1]])


@pytest.mark.parametrize("grid_m,grid_s", [(7, 1), (40, 3), (200, 5), (33, 16)])
def test_ragged_grids(gpu, oracle, grid_m, grid_s):
    cl = synth.Cluster(np.array([8, 4, 4, 2, 1, 0], np.int16))      # heterogeneous nodes
    jobs = synth.draw_jobs(11, 21, grid_m, 16, cl.k_max)
    jobs = with_fair_share(jobs, cl)
    gp, sp, am = _gpu_table(gpu, cl, jobs, grid_s)
    gp_r, sp_r, am_r = oracle.build_speedup_table(jobs, cl.node_capacity, cl.k_max, cl.n_max, grid_s)
    check_table(oracle, jobs, grid_s, gp, sp, am, gp_r, sp_r, am_r)


def test_degenerate_jobs(gpu, oracle):
    cl = synth.uniform_cluster(4, 4)
    jobs = synth.draw_jobs(6, 3, 32, 8, cl.k_max)
    # prior-driven exploration (Sec. 4.1): unexplored sync parameters are zero
    jobs.alpha_local[0] = jobs.beta_local[0] = 0.0
    jobs.beta_local[1] = jobs.beta_node[1] = 0.0
    jobs.alpha_local[2] = jobs.beta_local[2] = jobs.alpha_node[2] = jobs.beta_node[2] = 0.0
    jobs.gamma[3] = 1.0
    jobs.gamma[4] = 10.0
    jobs.m_max_total[5] = jobs.m0[5]            # only M = M0 is allowed: many (K, N) infeasible
    jobs = with_fair_share(jobs, cl)
    gp, sp, am = _gpu_table(gpu, cl, jobs, 8)
    gp_r, sp_r, am_r = oracle.build_speedup_table(jobs, cl.node_capacity, cl.k_max, cl.n_max, 8)
    check_table(oracle, jobs, 8, gp, sp, am, gp_r, sp_r, am_r)
    assert (gp_r[5] == 0).sum() > (gp_r[0] == 0).sum()


def test_invalid_fair_share_and_optional_outputs(gpu, oracle):
    cl = synth.uniform_cluster(4, 4)
    jobs = synth.draw_jobs(5, 4, 32, 8, cl.k_max)
    jobs = with_fair_share(jobs, cl, fair=(3, 1))
    jobs.fair_k[1], jobs.fair_n[1] = 9, 1         # does not fit one node: no denominator
    jobs.fair_k[2], jobs.fair_n[2] = 500, 700     # outside the table
    jobs.fair_k[3], jobs.fair_n[3] = -1, -1
    gp, sp, am = _gpu_table(gpu, cl, jobs, 8, want_goodput=False, want_argmax=False)
    assert gp is None and am is None
    gp_r, sp_r, am_r = oracle.build_speedup_table(jobs, cl.node_capacity, cl.k_max, cl.n_max, 8)
    assert_close(sp, sp_r, what="speedup")
    assert not sp[1].any() and not sp[2].any() and not sp[3].any() and sp[0].any()


def test_single_job_and_custom_dims(gpu, oracle):
    cl = synth.uniform_cluster(3, 8)
    jobs = with_fair_share(synth.draw_jobs(1, 9, 32, 8, 24), cl)
    gp, sp, am = _gpu_table(gpu, cl, jobs, 8, k_max=20, n_max=2)
    gp_r, sp_r, am_r = oracle.build_speedup_table(jobs, cl.node_capacity, 20, 2, 8)
    assert gp.shape == (1, 21, 3)
    check_table(oracle, jobs, 8, gp, sp, am, gp_r, sp_r, am_r)


@pytest.mark.parametrize("grid_m,grid_s,case", [(1, 8, ""), (3, 32, ""), (128, 9, "flat"), (129, 4, "flat"), (300, 3, ""),
                                                (1030, 2, ""), (64, 8, "big"), (16, 200, "steps")])
def test_screened_sweep_edges(gpu, oracle, grid_m, grid_s, case):
    """Lengths of the grid around what a thread and a block can screen, jobs whose goodput hardly
    depends on m (dozens of points within the screening margin), batch sizes beyond the screening's
    exact quotients, many accumulation steps; slabs of a width that is no multiple of four."""
    cl = synth.Cluster(np.array([8, 8, 4, 4, 2], np.int16))
    jobs = synth.draw_jobs(5, 33, grid_m, max(grid_s, 8), cl.k_max)
    if case == "flat":
        jobs.alpha_grad[:] = 1e-6
        jobs.alpha_local[:] = jobs.alpha_node[:] = 1e-7
        jobs.beta_local[:] = jobs.beta_node[:] = 0.0
        jobs.phi[:] = 1e6
    if case == "big":
        jobs.m0[:] = 1 << 20
        jobs.m_max_total[:] = 12 << 20
        jobs.m_max_gpu[:] = 1 << 18
        jobs.m_grid = synth.make_m_grid(jobs.m_max_gpu, grid_m)
    jobs = with_fair_share(jobs, cl)
    gp, sp, am = _gpu_table(gpu, cl, jobs, grid_s, k_max=14, n_max=4)
    gp_r, sp_r, am_r = oracle.build_speedup_table(jobs, cl.node_capacity, 14, 4, grid_s)
    check_table(oracle, jobs, grid_s, gp, sp, am, gp_r, sp_r, am_r)


@pytest.mark.parametrize("nodes,gpus,jobs", [(32, 1, 300), (17, 4, 300), (28, 8, 60), (9, 8, 150), (50, 1, 300), (22, 4, 1000),
                                             (6, 2, 37), (16, 4, 48)])
def test_slabs_of_any_width_and_place(gpu, oracle, nodes, gpus, jobs):
    """A slab's fours of entries are aligned in the whole table, so a thread's first one may begin before the
    slab; widths at which its next ones would still be counted from there, and others."""
    cl = synth.uniform_cluster(nodes, gpus)
    j = with_fair_share(synth.draw_jobs(jobs, 5, 32, 8, cl.k_max), cl)
    gp, sp, am = _gpu_table(gpu, cl, j, 8)
    gp_r, sp_r, am_r = oracle.build_speedup_table(j, cl.node_capacity, cl.k_max, cl.n_max, 8)
    check_table(oracle, j, 8, gp, sp, am, gp_r, sp_r, am_r)


@pytest.mark.parametrize("kind,nodes,gpus,points,steps,many,few", [
    ("grid", 4, 4, 32, 16, 900, 7), ("grid", 6, 2, 100, 8, 2500, 30), ("grid", 17, 4, 64, 16, 400, 21), ("grid", 32, 8, 128, 32, 100, 24),
    ("grid", 4, 4, 300, 8, 3000, 40), ("grid", 1, 1, 33, 8, 9000, 3), ("flat", 6, 4, 128, 9, 900, 20), ("flat", 6, 4, 129, 4, 5000, 20),
    ("big", 5, 8, 64, 8, 500, 11), ("samples", 8, 4, 48, 1, 400, 20), ("samples", 5, 8, 128, 1, 700, 50),
    ("samples", 3, 2, 300, 1, 9000, 9), ("fixed", 8, 4, 90, 1, 600, 20), ("rack", 9, 8, 64, 16, 200, 12), ("rack", 4, 4, 31, 8, 2000, 5)])
def test_tables_in_two_launches_equal_those_in_one(gpu, oracle, kind, nodes, gpus, points, steps, many, few):
    """Few (job, K, class): a sweep of all points and the slabs, two launches; many: one launch that screens.  The
    same job's table is the same bit for bit, and a sample agrees with the oracle."""
    torch, api = gpu
    cl = synth.uniform_cluster(nodes, gpus)
    samples = kind in ("samples", "fixed")
    jobs = synth.draw_jobs(many, 5, 32 if samples else points, max(steps, 8), cl.k_max)
    if kind == "flat":
        jobs.alpha_grad[:] = 1e-6
        jobs.alpha_local[:] = jobs.alpha_node[:] = 1e-7
        jobs.beta_local[:] = jobs.beta_node[:] = 0.0
        jobs.phi[:] = 1e6
    if kind == "big":
        jobs.m0[:] = 1 << 20
        jobs.m_max_total[:] = 12 << 20
        jobs.m_max_gpu[:] = 1 << 18
        jobs.m_grid = synth.make_m_grid(jobs.m_max_gpu, points)
    jobs = with_fair_share(jobs, cl)
    adaptive = (np.arange(many) % 3 != 0).astype(np.uint8) if kind == "fixed" else None
    ar, br = synth.draw_rack_pair(jobs, 8)
    idx = np.unique(np.linspace(0, many - 1, few).astype(int))
    out = []
    for take, launches in ((np.arange(many), 1), (idx, 2)):
        j = jobs.take(take)
        dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
        s = api.Scheduler(node_capacity=cl.node_capacity, num_jobs=j.num_jobs, grid_m=j.m_grid.shape[1], grid_s=max(steps, 1),
                          population=1, stream=torch.cuda.current_stream().cuda_stream)
        dj = api.DeviceJobs(j, "cuda", torch)
        gp = torch.full(s.table_shape, -1.0, device="cuda")
        sp, am = torch.full_like(gp, -1.0), torch.full(s.table_shape, 7, dtype=torch.uint16, device="cuda")
        s.set_kernel_timing(True)
        if samples:
            s.build_speedup_table_msample(dj, dev(synth.make_m_samples(j.m0, j.m_max_total, points)), dev(j.m_max_gpu), gp, sp, am,
                                          adaptive=None if adaptive is None else dev(adaptive[take]))
        elif kind == "rack":
            s.build_speedup_table_rack(dj, dev(ar[take]), dev(br[take]), gp, sp, am)
        else:
            s.build_speedup_table(dj, gp, sp, am)
        s.sync_status()
        assert s.read_kernel_timing()["speedup_table"][1] == launches
        out.append([x.cpu().numpy() for x in (gp, sp, am)])
        s.close()
    for one, two in zip(*out):
        assert np.array_equal(one[idx], two)
    if kind in ("grid", "flat", "big"):
        ref = oracle.build_speedup_table(jobs.take(idx), cl.node_capacity, cl.k_max, cl.n_max, steps)
        check_table(oracle, jobs.take(idx), steps, *out[1], *ref)
    assert (out[0][0] > 0).any()
