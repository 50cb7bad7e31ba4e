"""Throughput-model fitting (Sec. 4.1): pins of the oracle's objective and CUDA parity on the
objective value and on the quality of the minimiser."""
import numpy as np
import pytest

from paper_2008_12260_b200 import synth


def _fit():
    from oracle import fit
    return fit


def test_objective_closed_forms():
    fit = _fit()
    th = [1.0, 0.02, 4.0, 0.0, 9.0, 0.5, 2.0]
    # T_grad = 3, local sync 4, gamma 2 -> 5; two accumulation steps -> 11 (Eq. 8-11)
    assert fit.t_iter(th, [4], [1], [100], [2])[0] == pytest.approx(11.0, rel=1e-14)
    # node pair with retrogression: 9 + 0.5 * (6 - 2) = 11; T_grad = 3 -> sqrt(9 + 121)
    assert fit.t_iter(th, [6], [2], [100], [0])[0] == pytest.approx(130 ** 0.5, rel=1e-14)
    # one replica: no synchronisation; gamma = 1: plain sum
    assert fit.t_iter(th, [1], [1], [100], [3])[0] == pytest.approx(12.0, rel=1e-14)
    th1 = th[:6] + [1.0]
    assert fit.t_iter(th1, [4], [1], [100], [0])[0] == pytest.approx(7.0, rel=1e-14)
    # the error is 0 on exact data, and ln(1+2x) - ln(1+x) for a doubled prediction
    K, N, m, s = [4, 6, 1], [1, 2, 1], [100, 100, 100], [2, 0, 3]
    T = fit.t_iter(th, K, N, m, s)
    assert fit.rmsle(th, K, N, m, s, T) == 0.0
    assert fit.rmsle(th, [4], [1], [100], [2], [5.5]) == pytest.approx(np.log(12.0) - np.log(6.5), rel=1e-14)
    assert fit.rmsle(th, [], [], [], [], []) == 0.0


def test_oracle_fit_recovers_the_noise_floor():
    fit = _fit()
    rng = np.random.default_rng(0)
    true = np.array([0.05, 0.002, 0.02, 0.001, 0.06, 0.004, 3.0])
    n = 80
    K = rng.integers(1, 17, n); N = np.where(K == 1, 1, np.minimum(rng.integers(1, 5, n), K))
    m = rng.integers(8, 257, n); s = rng.integers(0, 4, n)
    T = fit.t_iter(true, K, N, m, s) * np.exp(rng.normal(0, 0.02, n))
    th0 = np.array([0.1, 0.01, 0.01, 0.01, 0.01, 0.01, 1.0])
    x, f = fit.fit(K, N, m, s, T, th0)
    assert f <= fit.rmsle(true, K, N, m, s, T) * 1.05 and f < fit.rmsle(th0, K, N, m, s, T) / 10
    assert np.all(x[:6] >= 0) and 1.0 <= x[6] <= 10.0
    # frozen parameters stay where they were (prior-driven exploration keeps sync terms at 0)
    th0z = th0.copy(); th0z[2:6] = 0.0
    xz, fz = fit.fit(K, N, m, s, T, th0z, frozen=0b0111100)
    assert np.all(xz[2:6] == 0.0) and fz >= f * 0.999


DIVIDE = r"""
#include <stdio.h>
#include <stdint.h>
#include <string.h>
#include "divide.cuh"

static uint64_t state = 12345;
static uint64_t next64() {                       // splitmix64
  uint64_t z = (state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static double number(uint64_t bits, int exponent) {    // significand: random, or one where rounding is close
  uint64_t f = next64() & 0xFFFFFFFFFFFFFull;
  if (bits % 4 == 1) f = 0xFFFFFFFFFFFFFull - (next64() & 7);
  if (bits % 4 == 2) f = next64() & 7;
  if (bits % 4 == 3) f = (next64() & 7) << 49 | (next64() & 3);
  const double v = ldexp(1.0 + ldexp((double)f, -52), exponent);
  return bits & 64 ? -v : v;
}
int main() {
  long long n = 0, bad = 0;
  for (int k = 0; k < 20000000; ++k) {
    const uint64_t r = next64();
    int ea, eb;
    do {
      ea = -968 + (int)(next64() % 1988);
      eb = -1021 + (int)(next64() % 2041);
      if (r & 128) { ea = -40 + ea % 40; eb = -40 + eb % 40; }      // the usual exponents
    } while (ea - eb < -1019 || ea - eb > 1019);
    const double b = number(r >> 10, eb), a = k % 1000 ? number(r >> 20, ea) : 0.0, q = a / b, got = divide_by(a, b, 1.0 / b);
    ++n;
    bad += q != got;
  }
  printf("%lld %lld\n", n, bad);
  return 0;
}
"""


def test_division_by_a_reciprocal_is_the_division(tmp_path):
    """The quotient of two corrected multiplications equals the division's, bit for bit, over the exponents
    the method is stated for (fma and reciprocal are correctly rounded here as on the GPU)."""
    import subprocess
    from paper_2008_12260_b200 import build
    src, exe = tmp_path / "divide.cpp", tmp_path / "divide"
    src.write_text(DIVIDE)
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-I", build.CSRC, "-o", str(exe), str(src)])
    n, bad = subprocess.check_output([str(exe)]).split()
    assert int(n) == 20000000 and int(bad) == 0


def _problem(J, per_job, seed):
    fit = _fit()
    jobs = synth.draw_jobs(J, seed, 8, 4, 16)
    offset, K, N, m, s, factor = synth.draw_observations(jobs, per_job, seed + 1)
    true = np.stack([jobs.alpha_grad, jobs.beta_grad, jobs.alpha_local, jobs.beta_local, jobs.alpha_node,
                     jobs.beta_node, jobs.gamma], axis=1).astype(np.float64)
    T = np.empty(offset[-1], np.float32)
    for j in range(J):
        sl = slice(offset[j], offset[j + 1])
        T[sl] = (fit.t_iter(true[j], K[sl], N[sl], m[sl], s[sl]) * factor[sl]).astype(np.float32)
    theta0 = np.tile(np.array([0.1, 0.01, 0.01, 0.01, 0.01, 0.01, 1.0], np.float32), (J, 1))
    return fit, offset, K, N, m, s, T, theta0, true


@pytest.mark.gpu
def test_cuda_fit_against_oracle():
    import torch
    from paper_2008_12260_b200 import api

    J = 24
    per_job = np.array([0, 1, 3, 7] + [40 + 3 * i for i in range(J - 4)])
    fit, offset, K, N, m, s, T, theta0, true = _problem(J, per_job, 11)
    frozen = np.zeros(J, np.uint8)
    frozen[5] = 0b0111100; theta0[5, 2:6] = 0.0           # unexplored job: sync terms pinned at 0
    frozen[6] = 0b1000000; theta0[6, 6] = 2.5              # gamma pinned
    sch = api.Scheduler(node_capacity=np.full(4, 4, np.int16), num_jobs=1, grid_m=1, grid_s=1, population=1,
                        stream=torch.cuda.current_stream().cuda_stream)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    th_out = torch.zeros((J, 7), dtype=torch.float32, device="cuda")
    loss = torch.full((J,), -1.0, dtype=torch.float32, device="cuda")
    sch.fit_throughput_model(d(offset), d(K), d(N), d(m), d(s), d(T), d(theta0), th_out, loss, frozen=d(frozen),
                             max_iters=200)
    sch.sync_status()
    th_g, loss_g = th_out.cpu().numpy().astype(np.float64), loss.cpu().numpy().astype(np.float64)
    for j in range(J):
        sl = slice(offset[j], offset[j + 1])
        args = (K[sl], N[sl], m[sl], s[sl], T[sl])
        # 1. the reported error is the oracle's objective at the returned parameters
        assert loss_g[j] == pytest.approx(fit.rmsle(th_g[j], *args), rel=2e-4, abs=2e-6)
        # 2. bounds and frozen parameters
        assert np.all(th_g[j, :6] >= 0) and 1.0 <= th_g[j, 6] <= 10.0
        for i in range(7):
            if (frozen[j] >> i) & 1:
                assert th_g[j, i] == np.float32(theta0[j, i])
        # 3. as good a minimiser as L-BFGS-B from the same start
        _, f_ref = fit.fit(*args, theta0[j], frozen=int(frozen[j]))
        assert loss_g[j] <= f_ref * 1.05 + 2e-4, (j, loss_g[j], f_ref)
        if per_job[j] >= 40 and not frozen[j]:
            assert loss_g[j] < 0.05                       # near the 2 % noise floor
    assert loss_g[0] == 0.0 and np.array_equal(th_g[0].astype(np.float32), theta0[0])   # no observations
    sch.close()
