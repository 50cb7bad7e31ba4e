// Batched fitting of the throughput-model parameters theta_sys (Sec. 4.1, "online model
// fitting"): for every job, minimise the root mean squared logarithmic error between
// Eq. 11 and the observed (a, m, s, T_iter) tuples, with alpha, beta >= 0 and gamma in
// [1, 10].  The paper uses L-BFGS-B on one CPU core per job; here one block fits one job with a
// projected Levenberg-Marquardt iteration in double precision.
//
// A fit is a chain of dependent steps (solve, evaluate, accept), some fifty of them, so its length is
// what counts, not the arithmetic: of 1024 jobs x 64 observations most need some 15 steps, one needs 190, and
// that one is the time of the call.  Per step:
//  * the residual and its derivatives come from one logarithm of the ratio of the two times, with two
//    exponentials and a log1p, instead of five powers;
//  * a trial point is evaluated with its normal equations, so that an accepted one needs no second pass;
//  * the normal equations have 32 sums (a row of observations never has both synchronisation pairs): a
//    reduce-scatter leaves one per lane after 31 exchanges, in place of five for each sum;
//  * the 7 x 7 system is solved by all lanes alike, in registers, unrolled;
//  * two pairs of warps try two dampings at once (the one wanted, and the one wanted if that is
//    rejected, as nearly every second is): the first of the two that lowers the error is taken, as one
//    after the other would have it.
// Measured for 1024 jobs x 64 observations: 0.65 ms (2.9 - 3.1 ms with one trial at a time, powers and a pass per sum).
#include "common.cuh"

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

// T_iter of Eq. 11 and its derivatives: with hi the larger of T_grad and T_sync and x = (lo / hi)^gamma,
// the overlap is hi (1 + x)^(1 / gamma).
struct Model {
  double p;                // T_iter
  double d_tg, d_ts, d_g;  // of p, by T_grad, T_sync and gamma
};
__device__ __forceinline__ Model t_iter_model(double tg, double ts, double g, double inv_g, double s) {
  Model o;
  double ov = tg, e_tg = 1.0;
  o.d_ts = 0.0;
  o.d_g = 0.0;
  if (ts > 0.0 && tg > 0.0) {
    const bool grad_first = tg >= ts;
    const double hi = grad_first ? tg : ts, lo = grad_first ? ts : tg;
    const double r = lo / hi, lr = log(r), x = exp(g * lr), l1 = log1p(x), lg = l1 * inv_g;
    const double E = exp(lg), q = 1.0 / (1.0 + x);
    const double d_hi = E * q, d_lo = r > 0.0 ? d_hi * x / r : 0.0;
    ov = hi * E;
    e_tg = grad_first ? d_hi : d_lo;
    o.d_ts = grad_first ? d_lo : d_hi;
    o.d_g = ov * ((x > 0.0 ? x * lr * q : 0.0) - lg) * inv_g;
  } else if (ts > 0.0) {   // tg == 0
    ov = ts;
    e_tg = 0.0;
    o.d_ts = 1.0;
  }
  o.p = s * tg + ov;
  o.d_tg = s + e_tg;
  return o;
}

constexpr int PAIR = 64;         // threads that evaluate one trial
constexpr int TRIALS = 2;        // trials evaluated at once

// The 32 sums at `th` over the observations of this warp's half of the pair into out[0 .. 31] (shared).
__device__ __noinline__ void evaluate(const FitArgs &a, int lo, int hi, const double *th, const double *s_lt, double *out, int at) {
  const int lane = at & 31;
  double v[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = 0.0;
  const double t0 = th[0], t1 = th[1], t2 = th[2], t3 = th[3], t4 = th[4], t5 = th[5], g = th[6], inv_g = 1.0 / g;
#pragma unroll 1
  for (int o = lo + at; o < hi; o += PAIR) {
    const int K = __ldg(a.k + o), N = __ldg(a.n + o);
    const double m = (double)__ldg(a.m + o), s = (double)__ldg(a.s + o), k2 = (double)(K - 2);
    const double lt = o - lo < FIT_CACHE ? s_lt[o - lo] : log1p((double)a.t[o]);
    const bool sync = K >= 2, local = sync && N == 1;
    const double ts = sync ? (local ? t2 + t3 * k2 : t4 + t5 * k2) : 0.0;
    const Model f = t_iter_model(t0 + t1 * m, ts, g, inv_g, s);
    const double r = log1p(f.p) - lt, w = 1.0 / (1.0 + f.p);
    const double j_s = f.d_ts * w, j_k = j_s * k2;
    double j[NP];
    j[0] = f.d_tg * w;
    j[1] = j[0] * m;
    j[2] = local ? j_s : 0.0;
    j[3] = local ? j_k : 0.0;
    j[4] = sync && !local ? j_s : 0.0;
    j[5] = sync && !local ? j_k : 0.0;
    j[6] = f.d_g * w;
#pragma unroll
    for (int x = 0; x < NP; ++x) {
#pragma unroll
      for (int y = x; y < NP; ++y)
        if (sum_of(x, y) >= 0) v[sum_of(x, y) >= 0 ? sum_of(x, y) : 0] += j[x] * j[y];
      v[SUM_G + x] += j[x] * r;
    }
    v[SUM_S] += r * r;
  }
  // reduce-scatter: lane l is left with sum l (each sum over the lanes in the order of a xor tree)
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < off; ++i) {
      const double keep = upper ? v[i + off] : v[i], give = upper ? v[i] : v[i + off];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
    }
  }
  out[lane] = v[0];
}

// The damped step (A + lambda diag(A) + eps) d = -g on the free parameters, by Cholesky; 0 when the
// matrix is not positive definite.  All lanes work it out alike.
__device__ __noinline__ void solve(const double *sums, unsigned free_, double lambda, double (&d)[NP]) {
  double L[NP][NP], inv[NP];
  bool ok = true;
#pragma unroll
  for (int x = 0; x < NP; ++x) {
    const bool fx = (free_ >> x) & 1u;
#pragma unroll
    for (int y = 0; y <= x; ++y) {
      const int at = sum_of(y, x);
      double sum = at >= 0 && fx && ((free_ >> y) & 1u) ? sums[at >= 0 ? at : 0] : 0.0;
      if (x == y) sum = fx ? sum * (1.0 + lambda) + 1e-30 : 1.0;
#pragma unroll
      for (int z = 0; z < y; ++z) sum -= L[x][z] * L[y][z];
      if (x == y) {
        ok = ok && sum > 0.0;
        inv[x] = rsqrt(sum);
      } else {
        L[x][y] = sum * inv[y];
      }
    }
    d[x] = fx ? -sums[SUM_G + x] : 0.0;
  }
#pragma unroll
  for (int x = 0; x < NP; ++x) {             // forward, then backward substitution
    double sum = d[x];
#pragma unroll
    for (int z = 0; z < x; ++z) sum -= L[x][z] * d[z];
    d[x] = sum * inv[x];
  }
#pragma unroll
  for (int x = NP - 1; x >= 0; --x) {
    double sum = d[x];
#pragma unroll
    for (int z = x + 1; z < NP; ++z) sum -= L[z][x] * d[z];
    d[x] = sum * inv[x];
  }
#pragma unroll
  for (int x = 0; x < NP; ++x) d[x] = ok ? d[x] : 0.0;
}

// Three blocks of an SM: a fourth would spill (0.70 ms), two wait more (no faster).
__global__ void __launch_bounds__(PAIR * TRIALS, 3) fit_kernel(const __grid_constant__ FitArgs a) {
  // sums of the two halves of each trial's pair; sums at th; trial points
  __shared__ double s_lt[FIT_CACHE], s_part[TRIALS][2][32], s_sums[32], s_th[TRIALS][NP];
  const int tid = threadIdx.x, lane = tid & 31, j = blockIdx.x;
  const int trial = tid / PAIR, at = tid & (PAIR - 1);
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
    for (int i = tid; i < min(n, FIT_CACHE); i += PAIR * TRIALS) s_lt[i] = log1p((double)a.t[lo + i]);
    // the trial's point is laid down and evaluated by its pair of warps
    auto evaluate_at = [&](const double (&x)[NP]) {
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if (at == i) s_th[trial][i] = x[i];
      __syncthreads();
      evaluate(a, lo, hi, s_th[trial], s_lt, s_part[trial][at >> 5], at);
      __syncthreads();
    };
    auto take_sums = [&](int t) {            // the sums of a trial become those at th
      if (tid < 32) s_sums[lane] = s_part[t][0][lane] + s_part[t][1][lane];
      __syncthreads();
    };
    double d[NP];
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
        if (it >= 0) solve(s_sums, free_, trial ? lambda * 4.0 : lambda, d);
#pragma unroll
        for (int i = 0; i < NP; ++i) d[i] = it >= 0 ? fmin(fmax(th[i] + d[i], lb[i]), ub[i]) : th[i];
        evaluate_at(d);
        double Sc = s_part[0][0][SUM_S] + s_part[0][1][SUM_S];
        if (it < 0) {                         // the starting point
          S = Sc;
          take_sums(0);
          break;
        }
        int t = 0;
        if (!(Sc < S)) {
          t = 1;
          lambda *= 4.0;
          Sc = s_part[1][0][SUM_S] + s_part[1][1][SUM_S];
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
    fit_kernel<<<num_jobs, PAIR * TRIALS, 0, ctx->stream>>>(a);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}
