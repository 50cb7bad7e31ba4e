// Batched fitting of the throughput-model parameters theta_sys (Sec. 4.1, "online model
// fitting"): for every job, minimise the root mean squared logarithmic error between
// Eq. 11 and the observed (a, m, s, T_iter) tuples, with alpha, beta >= 0 and gamma in
// [1, 10].  The paper uses L-BFGS-B on one CPU core per job; here one block fits one job with a
// projected Levenberg-Marquardt iteration in double precision.
//
// A fit is a chain of dependent steps (solve, evaluate, accept), some fifty of them, so its length is
// what counts, not the arithmetic: of 1024 jobs x 64 observations most need some 15 steps, one needs 190, and
// that one is the time of the call.  Where observations leave a parameter open, what it ends at hangs on the
// last bit of every step, so the arithmetic and the order of every sum are those of one warp taking one step
// after the other; what is shorter is the way there:
//  * two threads share an observation (the powers of T_grad and those of T_sync), three powers deep, not five;
//  * a trial point is evaluated with its normal equations, so that an accepted one needs no second pass;
//  * the normal equations have 32 sums (an observation never has both synchronisation pairs): the four warps
//    of a trial take eight each, and a reduce-scatter leaves one per lane after nine exchanges, in place of
//    five for each sum; its tree adds the same pairs in the same order;
//  * the 7 x 7 system is solved in registers, unrolled, with one reciprocal per column;
//  * two groups of warps try two dampings at once (the one wanted, and the one wanted if that is
//    rejected, as nearly every second is): the first of the two that lowers the error is taken, as one
//    after the other would have it.
// Measured for 1024 jobs x 64 observations: 1.06 ms (3.1 ms with one warp taking one step after the other).
#include "common.cuh"
#include "divide.cuh"

namespace {

constexpr int NP = 7;   // alpha_grad, beta_grad, alpha_local, beta_local, alpha_node, beta_node, gamma
constexpr int FIT_CACHE = 128;   // observations per job whose ln(1 + T) is kept

struct FitArgs {
  const int32_t *offset;   // [J + 1] observations of job j are offset[j] .. offset[j + 1]
  const int32_t *k, *n, *m, *s;
  const float *t;
  const float *theta0;     // [J][7]
  const uint8_t *frozen;   // [J] bit i set: parameter i is held at its starting value, or NULL
  int J, max_iters;
  float *theta_out;        // [J][7]
  float *loss_out;         // [J]
};

// Place of A[x][y], x <= y, of the normal equations among the sums; -1: always zero (a local and a
// node parameter).  Then the seven of the gradient, then the sum of squares.
__host__ __device__ constexpr int sum_of(int x, int y) {
  if (x >= 2 && x <= 3 && y >= 4 && y <= 5) return -1;
  int at = 0;
  for (int i = 0; i < x; ++i) at += (NP - i) - ((i == 2 || i == 3) ? 2 : 0);
  at += y - x;
  if ((x == 2 || x == 3) && y > 5) at -= 2;
  return at;
}
constexpr int SUM_G = 24, SUM_S = 31;
static_assert(sum_of(6, 6) == 23, "24 products, 7 gradients, 1 square");

constexpr int TILE = 64;             // observations at a time
constexpr int GROUP = 2 * TILE;      // threads that evaluate one trial
constexpr int TRIALS = 2;            // trials evaluated at once

// What an observation adds to the sums is made of these: the derivatives of T_iter (Eq. 11) by T_grad,
// by T_sync and by gamma, 1 / (1 + T_iter), the residual.
struct Observed {
  double d_tg[TILE], d_ts[TILE], d_g[TILE], w[TILE], r[TILE], m[TILE], k2[TILE];
  int pair[TILE];                    // 0: local pair, 1: node pair, -1: none
};

// Place of the x-th factor: which parameters make sum `at` (7, 7 for the sum of squares; y = 7 for the gradient)
__host__ __device__ constexpr int sum_x(int at) {
  if (at == SUM_S) return 7;
  if (at >= SUM_G) return at - SUM_G;
  for (int x = 0; x < NP; ++x)
    for (int y = x; y < NP; ++y)
      if (sum_of(x, y) == at) return x;
  return -1;
}
__host__ __device__ constexpr int sum_y(int at) {
  if (at >= SUM_G) return 7;
  for (int x = 0; x < NP; ++x)
    for (int y = x; y < NP; ++y)
      if (sum_of(x, y) == at) return y;
  return -1;
}

template <int AT>
__device__ __forceinline__ void add_one(const double (&grad)[NP], double w, double r, double &v) {
  constexpr int x = sum_x(AT), y = sum_y(AT);
  if constexpr (AT == SUM_S) {
    v = fma(r, r, v);
  } else if constexpr (y == 7) {
    v = fma(__dmul_rn(grad[x], w), r, v);
  } else {
    v = fma(__dmul_rn(__dmul_rn(grad[x], w), grad[y]), w, v);
  }
}

// Sums FIRST .. FIRST + 7: lane l adds observations l, l + 32, .. of the tile.
template <int FIRST>
__device__ __forceinline__ void add_observations(const Observed &ob, int lane, double (&v)[8]) {
#pragma unroll
  for (int o = lane; o < TILE; o += 32) {
    const double w = ob.w[o], r = ob.r[o], d_ts = ob.d_ts[o], d_tk = d_ts * ob.k2[o];
    const int pair = ob.pair[o];
    const double grad[NP] = {ob.d_tg[o], ob.d_tg[o] * ob.m[o], pair == 0 ? d_ts : 0.0, pair == 0 ? d_tk : 0.0,
                             pair == 1 ? d_ts : 0.0, pair == 1 ? d_tk : 0.0, ob.d_g[o]};
    add_one<FIRST + 0>(grad, w, r, v[0]);
    add_one<FIRST + 1>(grad, w, r, v[1]);
    add_one<FIRST + 2>(grad, w, r, v[2]);
    add_one<FIRST + 3>(grad, w, r, v[3]);
    add_one<FIRST + 4>(grad, w, r, v[4]);
    add_one<FIRST + 5>(grad, w, r, v[5]);
    add_one<FIRST + 6>(grad, w, r, v[6]);
    add_one<FIRST + 7>(grad, w, r, v[7]);
  }
}

// The 32 sums at `th` into out[0 .. 31] (shared), by the GROUP threads of a trial; at: which of them.
// The whole block calls it.
__device__ __noinline__ void evaluate(const FitArgs &a, int lo, int hi, const double *th, const double *s_lt, Observed &ob,
                                      double *out, int at) {
  const int lane = at & 31, warp = at >> 5, q = at >> 1;
  const bool sync_part = (at & 1) != 0;      // this thread has T_sync, its neighbour T_grad
  double v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = 0.0;
  const double t0 = th[0], t1 = th[1], t2 = th[2], t3 = th[3], t4 = th[4], t5 = th[5], g = th[6];
#pragma unroll 1
  for (int first = lo; first < hi; first += TILE) {
    const int o = first + q;
    const bool live = o < hi;
    const int K = live ? __ldg(a.k + o) : 1, N = live ? __ldg(a.n + o) : 1;
    const double m = live ? (double)__ldg(a.m + o) : 0.0, s = live ? (double)__ldg(a.s + o) : 0.0, k2 = (double)(K - 2);
    const int pair = K < 2 ? -1 : N == 1 ? 0 : 1;
    const double tg = t0 + t1 * m;
    const double ts = pair < 0 ? 0.0 : pair == 0 ? t2 + t3 * k2 : t4 + t5 * k2;
    const bool both = live && ts > 0.0 && tg > 0.0;
    const double mine = both ? (sync_part ? ts : tg) : 1.0;
    double ov = ts > 0.0 && !(tg > 0.0) ? ts : tg;
    double d_mine = ts > 0.0 && !(tg > 0.0) ? (sync_part ? 1.0 : 0.0) : (sync_part ? 0.0 : 1.0);
    double d_g = 0.0;
    if (__any_sync(0xffffffffu, both)) {
      const double pw = pow(mine, g), lg = log(mine);
      const double other = __shfl_xor_sync(0xffffffffu, pw, 1), lg_other = __shfl_xor_sync(0xffffffffu, lg, 1);
      const double pa = sync_part ? other : pw, pb = sync_part ? pw : other;
      const double la = sync_part ? lg_other : lg, lb = sync_part ? lg : lg_other;
      const double sum = pa + pb;
      const double over = pow(sum, 1.0 / g);
      const double dm = pow(mine / over, g - 1.0);
      if (both) {
        ov = over;
        d_mine = dm;
        if (sync_part) d_g = ov * (-log(sum) / (g * g) + (pa * la + pb * lb) / (g * sum));
      }
    }
    if (sync_part) {
      ob.d_ts[q] = live ? d_mine : 0.0;
      ob.d_g[q] = d_g;
      ob.k2[q] = k2;
      ob.m[q] = m;
      ob.pair[q] = pair;
    } else {
      const double p = s * tg + ov;
      ob.d_tg[q] = live ? s + d_mine : 0.0;
      ob.w[q] = live ? 1.0 / (1.0 + p) : 0.0;
      ob.r[q] = live ? log1p(p) - (o - lo < FIT_CACHE ? s_lt[o - lo] : log1p((double)a.t[o])) : 0.0;
    }
    __syncthreads();
    if (warp == 0) add_observations<0>(ob, lane, v);
    else if (warp == 1) add_observations<8>(ob, lane, v);
    else if (warp == 2) add_observations<16>(ob, lane, v);
    else add_observations<24>(ob, lane, v);
    if (first + TILE < hi) __syncthreads();
  }
  // reduce-scatter: lane l is left with sum l / 4 (each over the lanes in the order of a xor tree)
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const bool upper = (lane & off) != 0;
    if (off >= 4) {
#pragma unroll
      for (int i = 0; i < off / 4; ++i) {
        const double keep = upper ? v[i + off / 4] : v[i], give = upper ? v[i] : v[i + off / 4];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    }
  }
  if ((lane & 3) == 0) out[warp * 8 + (lane >> 2)] = v[0];
}

// The damped step (A + lambda diag(A) + eps) d = -g on the free parameters, by Cholesky; 0 when the
// matrix is not positive definite.  All lanes of a warp work it out alike.
__device__ __noinline__ void solve(const double *sums, unsigned free_, double lambda, double (&d)[NP]) {
  double L[NP][NP], inv[NP];
  bool ok = true;
#pragma unroll
  for (int y = 0; y < NP; ++y) {              // column by column
#pragma unroll
    for (int x = y; x < NP; ++x) {
      const bool fx = (free_ >> x) & 1u;
      const int at = sum_of(y, x);
      double sum = at >= 0 && fx && ((free_ >> y) & 1u) ? sums[at >= 0 ? at : 0] : 0.0;
      if (x == y) sum = fx ? fma(sum, 1.0 + lambda, 1e-30) : 1.0;
#pragma unroll
      for (int z = 0; z < y; ++z) sum = fma(-L[x][z], L[y][z], sum);
      if (x == y) {
        ok = ok && !(sum <= 0.0);
        L[x][x] = sqrt(sum);
        inv[x] = 1.0 / L[x][x];
      } else {
        L[x][y] = divide_by(sum, L[y][y], inv[y]);
      }
    }
  }
#pragma unroll
  for (int x = 0; x < NP; ++x) {             // forward, then backward substitution
    double sum = (free_ >> x) & 1u ? -sums[SUM_G + x] : 0.0;
#pragma unroll
    for (int z = 0; z < x; ++z) sum = fma(-L[x][z], d[z], sum);
    d[x] = divide_by(sum, L[x][x], inv[x]);
  }
#pragma unroll
  for (int x = NP - 1; x >= 0; --x) {
    double sum = d[x];
#pragma unroll
    for (int z = x + 1; z < NP; ++z) sum = fma(-L[z][x], d[z], sum);
    d[x] = divide_by(sum, L[x][x], inv[x]);
  }
#pragma unroll
  for (int x = 0; x < NP; ++x) d[x] = ok ? d[x] : 0.0;
}

// Two blocks per SM: one leaves the short jobs waiting (1.35 ms), three spill (1.13 ms).
__global__ void __launch_bounds__(GROUP * TRIALS, 2) fit_kernel(const __grid_constant__ FitArgs a) {
  __shared__ double s_lt[FIT_CACHE], s_part[TRIALS][32], s_sums[32], s_th[TRIALS][NP];   // sums of the trials and at th
  __shared__ Observed s_obs[TRIALS];
  const int tid = threadIdx.x, j = blockIdx.x;
  const int trial = tid / GROUP, at = tid & (GROUP - 1);
  const int lo = a.offset[j], hi = a.offset[j + 1];
  const int n = hi - lo;
  const unsigned frozen = a.frozen ? a.frozen[j] : 0u;
  double th[NP], lb[NP], ub[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const double t0 = (double)a.theta0[(size_t)j * NP + i];
    lb[i] = (i == 6) ? 1.0 : 0.0;
    ub[i] = (i == 6) ? 10.0 : 1e300;
    th[i] = fmin(fmax(t0, lb[i]), ub[i]);
    if ((frozen >> i) & 1u) { th[i] = t0; lb[i] = ub[i] = t0; }
  }
  double S = 0.0;
  if (n > 0) {
#pragma unroll 1
    for (int i = tid; i < min(n, FIT_CACHE); i += GROUP * TRIALS) s_lt[i] = log1p((double)a.t[lo + i]);
    auto take_sums = [&](int t) {            // the sums of a trial become those at th
      if (tid < 32) s_sums[tid] = s_part[t][tid];
      __syncthreads();
    };
    double lambda = 1e-3;
#pragma unroll 1
    for (int it = -1; it < a.max_iters; ++it) {
      // free parameters: not frozen, and not sitting on a bound with the gradient pushing out
      unsigned free_ = 0u;
      if (it >= 0) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const double gi = s_sums[SUM_G + i];
          if (lb[i] < ub[i] && !((th[i] <= lb[i] && gi > 0.0) || (th[i] >= ub[i] && gi < 0.0))) free_ |= 1u << i;
        }
      }
      bool accepted = false;
#pragma unroll 1
      for (int tries = 0; tries < 8 && !accepted; tries += TRIALS) {
        if (at < 32) {                       // the trial's point
          double d[NP];
          if (it >= 0) solve(s_sums, free_, trial ? lambda * 4.0 : lambda, d);
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            const double x = it >= 0 ? fmin(fmax(th[i] + d[i], lb[i]), ub[i]) : th[i];
            if (at == i) s_th[trial][i] = x;
          }
        }
        __syncthreads();
        evaluate(a, lo, hi, s_th[trial], s_lt, s_obs[trial], s_part[trial], at);
        __syncthreads();
        double Sc = s_part[0][SUM_S];
        if (it < 0) {                         // the starting point
          S = Sc;
          take_sums(0);
          break;
        }
        int t = 0;
        if (!(Sc < S)) {
          t = 1;
          lambda *= 4.0;
          Sc = s_part[1][SUM_S];
        }
        if (Sc < S) {
          const double gain = (S - Sc) / fmax(S, 1e-300);
#pragma unroll
          for (int i = 0; i < NP; ++i) th[i] = s_th[t][i];
          S = Sc;
          lambda = fmax(lambda / 3.0, 1e-12);
          accepted = true;
          take_sums(t);
          if (gain < 1e-12) it = a.max_iters;           // converged
        } else {
          lambda *= 4.0;
          __syncthreads();                   // (the next trials' points take these ones' place)
        }
      }
      if (!accepted && it >= 0) break;
    }
  }
#pragma unroll
  for (int i = 0; i < NP; ++i)
    if (tid == i) a.theta_out[(size_t)j * NP + i] = (float)th[i];
  if (tid == 0) a.loss_out[j] = n > 0 ? (float)sqrt(S / (double)n) : 0.f;
}

}  // namespace

int launch_fit(sched_ctx *ctx, int32_t num_jobs, const int32_t *d_offset, const int32_t *d_k, const int32_t *d_n,
               const int32_t *d_m, const int32_t *d_s, const float *d_t, const float *d_theta0,
               const uint8_t *d_frozen, int32_t max_iters, float *d_theta_out, float *d_loss_out) {
  if (num_jobs == 0) return SCHED_OK;
  FitArgs a;
  a.offset = d_offset; a.k = d_k; a.n = d_n; a.m = d_m; a.s = d_s; a.t = d_t;
  a.theta0 = d_theta0; a.frozen = d_frozen; a.J = num_jobs; a.max_iters = max_iters;
  a.theta_out = d_theta_out; a.loss_out = d_loss_out;
  {
    TimedLaunch tl_(ctx, KK_FIT);
    fit_kernel<<<num_jobs, GROUP * TRIALS, 0, ctx->stream>>>(a);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}
