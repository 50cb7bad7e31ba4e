// Speedup-table builder: goodput sweep over the (m, s) grid (Eq. 4-11, 13) and
// normalisation by the fair-share goodput (Eq. 15): one launch per table, two for small ones.
//
// The goodput of an allocation depends on the allocation only through K = SUM(a) and its
// placement class (one node, several nodes, several racks; Eq. 9), so a job's sweep runs once
// per (K, class).  In one launch, a cluster of thread blocks serves one job: its blocks share the job's
// (K, class) pairs, every result goes to all of them (distributed shared memory), and each
// then writes its part of the job's [K][N] slabs from shared memory.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "fitness_common.cuh"

namespace cg = cooperative_groups;

namespace {

struct JobPtrs {
  const float *alpha_grad, *beta_grad, *alpha_local, *beta_local, *alpha_node, *beta_node;
  const float *alpha_rack, *beta_rack;
  const float *gamma, *phi, *m0, *m_max_total;
};

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (T_grad^g + T_sync^g)^(1/g) in ratio form: hi * (1 + (lo/hi)^g)^(1/g).  Both exponent
// arguments stay in [-inf, 1], so the approximate lg2/ex2 keep ~1e-7 relative accuracy.
__device__ __forceinline__ float overlap_time(float tg, float ts, float gamma, float inv_gamma) {
  if (ts <= 0.f) return tg;
  const float hi = fmaxf(tg, ts), lo = fminf(tg, ts);
  const float r = __fdividef(lo, hi);
  const float x = ex2_approx(gamma * lg2_approx(r));
  return __fmul_rn(hi, ex2_approx(lg2_approx(1.f + x) * inv_gamma));
}

__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }

// A candidate optimum: goodput = num / den; tie = (s << 16) | grid index (smaller wins).
struct Best {
  float num, den;
  uint32_t tie;
};

__device__ __forceinline__ bool beats(const Best &a, const Best &b) {
  const float l = a.num * b.den, r = b.num * a.den;
  return (l > r) || (l == r && a.num > 0.f && a.tie < b.tie);
}

__device__ __forceinline__ Best warp_best(Best best) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    Best o;
    o.num = __shfl_xor_sync(0xffffffffu, best.num, off);
    o.den = __shfl_xor_sync(0xffffffffu, best.den, off);
    o.tie = __shfl_xor_sync(0xffffffffu, best.tie, off);
    if (beats(o, best)) best = o;
  }
  return best;
}

// placement classes: a pair is K * 4 + class
enum { CLS_LOCAL = 0, CLS_NODE = 1, CLS_RACK = 2 };

struct TableArgs {
  JobPtrs jp;
  const int32_t *m_grid;        // [J][G] batch sizes per GPU (grid) or total batch sizes (samples)
  const int32_t *m_max_gpu;     // [J] (samples)
  const uint8_t *adaptive;      // [J] or NULL (samples)
  const int32_t *pairs;         // K * 4 + class: local and node pairs first, then rack pairs
  int pair_first, pair_count;   // the pairs of this launch
  const int32_t *kfit, *nmin, *fair_k, *fair_n;   // nmin: see TableRow
  int j_first, k_max, n_max, G, Gs;
  int parts, points;            // threads a (K, class) is shared by; G rounded up to equal stretches of fours (0: see MAX_POINTS)
  float *goodput, *speedup;     // [J][KD][ND] of the local and node classes (speedup NULL: not wanted)
  uint16_t *argmax;
  float *goodput_rack, *speedup_rack;   // the same of the rack class
  float one, zero;              // 1 and 0 (see grid_points)
  float *g;                     // [J][KD][3] results per (K, class) between the launches of a small table:
  uint16_t *a;                  // 0 and 0xFFFF where there is no such pair (nothing ever writes those)
  uint16_t *argmax_rack;
};

// A job's results per (K, class) in the shared memory of every block of its cluster.
struct TableSmem {
  float *g;        // [KD][3] goodput
  uint16_t *a;     // [KD][3] index of a maximiser
};

struct TableLayout {
  size_t g, a, point, best, multi, rows, total;
};
__host__ __device__ inline TableLayout table_layout(int KD, int points, int threads, int pairs) {
  TableLayout L;
  L.g = 0;
  L.a = L.g + (size_t)KD * 12;
  L.point = (L.a + (size_t)KD * 6 + 15) & ~(size_t)15;
  // (per screened point six floats; later a word per thread)
  L.best = L.point + (size_t)(points * 6 > threads ? points * 6 : threads) * 4;
  L.multi = L.best + (size_t)threads * 12;
  // the slab's rows take the place of everything but the results
  L.rows = L.point;
  const size_t end = L.multi + (size_t)pairs * 8, rows_end = L.rows + (size_t)(KD + 1) * 32;
  L.total = end > rows_end ? end : rows_end;
  return L;
}

// the job's parameters as the sweep uses them
struct JobModel {
  float a_g, b_g, gamma, inv_gamma, phi, M0, Mmax;
  float as[3], bs[3];      // synchronisation pair per class
};

__device__ __forceinline__ JobModel job_model(const JobPtrs &jp, int j) {
  JobModel m;
  m.a_g = jp.alpha_grad[j]; m.b_g = jp.beta_grad[j];
  m.gamma = jp.gamma[j]; m.inv_gamma = 1.f / m.gamma;
  m.phi = jp.phi[j]; m.M0 = jp.m0[j]; m.Mmax = jp.m_max_total[j];
  m.as[0] = jp.alpha_local[j]; m.bs[0] = jp.beta_local[j];
  m.as[1] = jp.alpha_node[j]; m.bs[1] = jp.beta_node[j];
  m.as[2] = jp.alpha_rack ? jp.alpha_rack[j] : 0.f; m.bs[2] = jp.beta_rack ? jp.beta_rack[j] : 0.f;
  return m;
}

__device__ __forceinline__ float sync_time(const JobModel &m, int K, int cls) {
  if (K < 2) return 0.f;
  const float a = cls == CLS_LOCAL ? m.as[0] : cls == CLS_NODE ? m.as[1] : m.as[2];
  const float b = cls == CLS_LOCAL ? m.bs[0] : cls == CLS_NODE ? m.bs[1] : m.bs[2];
  return fmaf(b, (float)(K - 2), a);
}

// a result to every block of the cluster
__device__ __forceinline__ void publish(cg::cluster_group &cl, const TableSmem &t, int at, float g, uint16_t a) {
  const unsigned n = cl.num_blocks();
  for (unsigned r = 0; r < n; ++r) {
    *cl.map_shared_rank(t.g + at, r) = g;
    *cl.map_shared_rank(t.a + at, r) = a;
  }
}

// integer range of u = s + 1 with M0 <= km u <= Mmax (products are exact integers below 2^24);
// qlo, qhi: approximate quotients M0 / km and Mmax / km - the four exact product tests correct an
// off-by-one in either direction
__device__ __forceinline__ void batch_window(float km, float M0, float Mmax, float qlo, float qhi, float gs, float &ulo,
                                             float &uhi) {
  ulo = ceilf(qlo);
  uhi = floorf(qhi);
  if (km * (ulo - 1.f) >= M0) ulo -= 1.f;
  if (km * ulo < M0) ulo += 1.f;
  if (km * (uhi + 1.f) <= Mmax) uhi += 1.f;
  if (km * uhi > Mmax) uhi -= 1.f;
  ulo = fmaxf(ulo, 1.f);
  uhi = fminf(uhi, gs);
}

// The best s of each of MQ grid points (m[q], index i + 32 q; only the first `count` of them exist), exactly
// as tabulated: with u = s + 1
//   T_iter = ta + u tg,  1/EFFICIENCY = c0 + u kr  (kr = K m / (phi + M0)),
//   goodput = K m * u / den(u),  den(u) = (ta + u tg)(c0 + u kr),
// the maximiser over ALL s by cross-multiplied compares (den(u)/u is convex in u, so goodput is
// unimodal in s), clamped into the window M0 <= K m u <= Mmax.  Several points go two by two through packed
// arithmetic, and what a compare chooses is moved by predicated multiply-adds with a one and a zero that the
// compiler does not know: compares and selects share the half-rate integer pipe (1024 jobs x 19 pairs x 300
// points: 67 us with plain selects, 63 us so).
template <int MQ>
__device__ __forceinline__ void grid_points(const JobModel &jm, float ts, float Kf, float rinv, float c0, const int (&m)[MQ],
                                            int i, int count, int Gs, float one, float zero, Best &best) {
  float tg[MQ], ta[MQ], kr[MQ], bu[MQ], bd[MQ];
#pragma unroll
  for (int q = 0; q < MQ; ++q) {
    tg[q] = fmaf(jm.b_g, (float)m[q], jm.a_g);
    ta[q] = __fsub_rn(overlap_time(tg[q], ts, jm.gamma, jm.inv_gamma), tg[q]);
    kr[q] = __fmul_rn(Kf * (float)m[q], rinv);
    bu[q] = 0.f;
    bd[q] = 1.f;
  }
  float u = 1.f;
#pragma unroll 4
  for (int s = 0; s < Gs; ++s, u += 1.f) {
    if (MQ == 1) {
      const float den = __fmul_rn(fmaf(u, tg[0], ta[0]), fmaf(u, kr[0], c0));
      if (__fmul_rn(u, bd[0]) > __fmul_rn(bu[0], den)) { bu[0] = u; bd[0] = den; }
    }
#pragma unroll
    for (int q = 0; q + 1 < MQ; q += 2) {
      const float2 u2 = f2(u);
      const float2 den = __fmul2_rn(__ffma2_rn(u2, make_float2(tg[q], tg[q + 1]), make_float2(ta[q], ta[q + 1])),
                                    __ffma2_rn(u2, make_float2(kr[q], kr[q + 1]), f2(c0)));
      const float2 l = __fmul2_rn(u2, make_float2(bd[q], bd[q + 1])), r = __fmul2_rn(make_float2(bu[q], bu[q + 1]), den);
      asm("{\n"
          " .reg .pred pa, pb;\n"
          " setp.gt.f32 pa, %4, %6;\n"
          " setp.gt.f32 pb, %5, %7;\n"
          " @pa fma.rn.f32 %0, %8, %11, %12;\n"
          " @pa fma.rn.f32 %2, %9, %11, %12;\n"
          " @pb fma.rn.f32 %1, %8, %11, %12;\n"
          " @pb fma.rn.f32 %3, %10, %11, %12;\n"
          "}"
          : "+f"(bu[q]), "+f"(bu[q + 1]), "+f"(bd[q]), "+f"(bd[q + 1])
          : "f"(l.x), "f"(l.y), "f"(r.x), "f"(r.y), "f"(u), "f"(den.x), "f"(den.y), "f"(one), "f"(zero));
    }
  }
#pragma unroll
  for (int q = 0; q < MQ; ++q) {
    const float km = Kf * (float)m[q], rkm = __frcp_rn(km);
    float ulo, uhi;
    batch_window(km, jm.M0, jm.Mmax, jm.M0 * rkm, jm.Mmax * rkm, (float)Gs, ulo, uhi);
    if (q >= count || !(ulo <= uhi)) continue;
    const float us = fminf(fmaxf(bu[q], ulo), uhi);
    Best b;
    b.num = km * us;
    b.den = (us == bu[q]) ? bd[q] : __fmul_rn(fmaf(us, tg[q], ta[q]), fmaf(us, kr[q], c0));
    b.tie = ((uint32_t)(us - 1.f) << 16) | (uint32_t)(i + 32 * q);
    if (beats(b, best)) best = b;
  }
}

// One grid point (a point of which no s is feasible is not scanned).
__device__ __noinline__ Best grid_point(const JobModel &jm, float ts, float Kf, float rinv, float c0, int m, int i,
                                        int Gs) {
  Best b = {0.f, 1.f, 0xFFFFFFFFu};
  const float mf = (float)m, km = Kf * mf;
  const float rkm = __frcp_rn(km);
  float ulo, uhi;
  batch_window(km, jm.M0, jm.Mmax, jm.M0 * rkm, jm.Mmax * rkm, (float)Gs, ulo, uhi);
  if (!(ulo <= uhi)) return b;
  const float tg = fmaf(jm.b_g, mf, jm.a_g);
  const float ta = __fsub_rn(overlap_time(tg, ts, jm.gamma, jm.inv_gamma), tg);
  const float kr = __fmul_rn(km, rinv);
  float bu = 0.f, bd = 1.f, u = 1.f;
#pragma unroll 4
  for (int s = 0; s < Gs; ++s, u += 1.f) {
    const float den = __fmul_rn(fmaf(u, tg, ta), fmaf(u, kr, c0));
    if (__fmul_rn(u, bd) > __fmul_rn(bu, den)) { bu = u; bd = den; }
  }
  const float us = fminf(fmaxf(bu, ulo), uhi);
  b.num = km * us;
  b.den = (us == bu) ? bd : __fmul_rn(fmaf(us, tg, ta), fmaf(us, kr, c0));
  b.tie = ((uint32_t)(us - 1.f) << 16) | (uint32_t)i;
  return b;
}

// The exact evaluation of one sampled total batch size M (Sec. 4.3): per_gpu = ceil(M / K), s =
// ceil(per_gpu / m_max) - 1 (the fewest accumulation steps that fit the per-GPU limit), m =
// ceil(per_gpu / (s + 1)); the batch actually run is M' = K m (s + 1), feasible when M0 <= M' <=
// M_max.  A non-adaptive job has the single candidate M0 and EFFICIENCY fixed to 1 (Sec. 4.2).
__device__ __forceinline__ Best sample_point_inline(const JobModel &jm, float ts, int K, float rinv, float c0, int mmax,
                                                    long long M, int i) {
  Best b = {0.f, 1.f, 0xFFFFFFFFu};
  if (M < 1) return b;
  long long s, m;
  if (M <= (1ll << 30)) {          // 32-bit divisions (the usual case) are several times cheaper
    const unsigned Mu = (unsigned)M, Ku = (unsigned)K, mu = (unsigned)mmax;
    const unsigned per_gpu = (Mu + Ku - 1u) / Ku;
    const unsigned su = (per_gpu + mu - 1u) / mu - 1u;
    s = su;
    m = (per_gpu + su) / (su + 1u);
  } else {
    const long long per_gpu = (M + K - 1) / K;
    s = (per_gpu + mmax - 1) / mmax - 1;
    m = (per_gpu + s) / (s + 1);
  }
  const float Mrun = (float)((long long)K * m * (s + 1));
  if (Mrun < jm.M0 || Mrun > jm.Mmax) return b;
  const float tg = fmaf(jm.b_g, (float)m, jm.a_g);
  const float tit = fmaf((float)s, tg, overlap_time(tg, ts, jm.gamma, jm.inv_gamma));
  b.num = Mrun;
  b.den = __fmul_rn(tit, fmaf(Mrun, rinv, c0));
  b.tie = (uint32_t)i;
  return b;
}

__device__ __noinline__ Best sample_point(const JobModel &jm, float ts, int K, float rinv, float c0, int mmax, long long M,
                                          int i) {
  return sample_point_inline(jm, ts, K, rinv, c0, mmax, M, i);
}

__device__ __forceinline__ bool kn_valid(int K, int N, int k_max, int n_max, const int32_t *__restrict__ kfit) {
  return N >= 1 && N <= n_max && K >= N && K <= k_max && K <= kfit[N];
}

// The job's slabs of (k_max + 1) x (n_max + 1) entries from its results per (K, class): broadcast
// along N, divided by the fair-share goodput (Eq. 15; one division per class, not per entry).  A row K of
// a slab holds one value at N = 1 and one from nmin[K] (the fewest nodes, two or more, that K replicas
// fit on) to K, so the rows are first laid down as such in shared memory (TableRow); the blocks of the
// cluster then write a piece of the slab each, in memory order, four entries at a time: aligned to 16
// bytes whatever the slab's width, a thread's (K, N) advancing without divisions.
struct TableRow {
  float sp1, sp2, g1, g2;      // N = 1, N >= 2
  int lo, hi;                  // nodes the second holds for
  uint32_t a12, pad;           // indices of the maximisers
};

__device__ __forceinline__ void write_slab(const TableRow *rows, int e0, int e1, size_t slab, int ND, float *speedup,
                                           float *goodput, uint16_t *argmax) {
  // entry e of the slab is entry slab + e of the whole table: fours are aligned there
  const int shift = (int)(slab & 3);
  const bool vec = (((uintptr_t)speedup | (uintptr_t)goodput) & 15) == 0 && ((uintptr_t)argmax & 7) == 0;
  const int step = (int)blockDim.x * 4, step_k = step / ND, step_n = step % ND;
  int e = (((e0 + shift) >> 2) + (int)threadIdx.x) * 4 - shift;     // may begin before e0
  int K = e < 0 ? 0 : e / ND, N = e < 0 ? e : e % ND;
  for (; e < e1; e += step) {
    float sp[4], g[4];
    uint32_t m[4];
    int k = K, n = N;
    TableRow r = rows[k];
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const bool many = n >= r.lo && n <= r.hi, one = n == 1;
      sp[z] = many ? r.sp2 : one ? r.sp1 : 0.f;
      g[z] = many ? r.g2 : one ? r.g1 : 0.f;
      m[z] = many ? r.a12 >> 16 : one ? r.a12 & 0xFFFFu : 0xFFFFu;
      if (++n == ND) { n = 0; ++k; r = rows[k]; }      // (one row more than the table has)
    }
    if (vec && e >= e0 && e + 4 <= e1) {
      *(float4 *)(speedup + slab + e) = make_float4(sp[0], sp[1], sp[2], sp[3]);
      if (goodput) *(float4 *)(goodput + slab + e) = make_float4(g[0], g[1], g[2], g[3]);
      if (argmax) *(uint2 *)(argmax + slab + e) = make_uint2(m[0] | (m[1] << 16), m[2] | (m[3] << 16));
    } else {
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        if (e + z < e0 || e + z >= e1) continue;
        speedup[slab + e + z] = sp[z];
        if (goodput) goodput[slab + e + z] = g[z];
        if (argmax) argmax[slab + e + z] = (uint16_t)m[z];
      }
    }
    K += step_k;
    N += step_n;
    if (N >= ND) { N -= ND; ++K; }
    else if (N < 0) { N += ND; --K; }       // (the thread's first four began before the slab)
  }
}

// where the job's fair-share goodput is (K * 3 + class), -1: there is none
__device__ __forceinline__ int fair_place(const TableArgs &a, int j) {
  const int kf = a.fair_k[j], nf = a.fair_n[j];
  return kn_valid(kf, nf, a.k_max, a.n_max, a.kfit) ? kf * 3 + (nf >= 2 ? CLS_NODE : CLS_LOCAL) : -1;
}

__device__ __forceinline__ void write_tables(const TableArgs &a, const TableSmem &t, TableRow *rows, int j, int rank, int nb,
                                             int fair) {
  const int KD = a.k_max + 1, ND = a.n_max + 1;
  const float denom = fair >= 0 ? t.g[fair] : 0.f;
  const int entries = KD * ND;
  const int e0 = (int)((long long)entries * rank / nb), e1 = (int)((long long)entries * (rank + 1) / nb);
#pragma unroll 1
  for (int rack = 0; rack < 2; ++rack) {
    if (!(rack ? a.speedup_rack : a.speedup)) continue;
    for (int K = threadIdx.x; K <= KD; K += blockDim.x) {
      TableRow r = {0.f, 0.f, 0.f, 0.f, 1, 0, 0xFFFFFFFFu, 0u};
      if (K < KD) {
        const int many = K * 3 + (rack ? CLS_RACK : CLS_NODE);
        if (!rack) { r.g1 = t.g[K * 3]; r.a12 = t.a[K * 3]; }
        else r.a12 = 0xFFFFu;
        r.g2 = t.g[many];
        r.a12 |= (uint32_t)t.a[many] << 16;
        if (denom > 0.f) { r.sp1 = r.g1 / denom; r.sp2 = r.g2 / denom; }
        r.lo = a.nmin[K];
        r.hi = min(K, a.n_max);
      }
      rows[K] = r;
    }
    __syncthreads();
    write_slab(rows, e0, e1, (size_t)j * entries, ND, rack ? a.speedup_rack : a.speedup, rack ? a.goodput_rack : a.goodput,
               rack ? a.argmax_rack : a.argmax);
    __syncthreads();
  }
}

// ---- the sweep ---------------------------------------------------------------------------------
// Tabulating a maximiser to the last bit needs the exact evaluation (grid_point: a scan over s;
// sample_point: integer divisions) at ONE point only, so all points are first screened: den(u)/u =
// A/u + B + C u has its real minimum at u* = sqrt(ta phi / (tg K m)), and the better of the two
// integers beside u* (clamped into the window) gives the point's goodput to about 1e-6, whatever the
// number of accumulation steps.  A thread screens the points of one (K, class) - or one of PARTS equal
// stretches of them, so that few jobs still fill the GPU - four at a time: what depends on m alone is in
// shared memory (one 16-byte broadcast each), the arithmetic is packed two by two, and rounding to an
// integer is an addition of 1.5 * 2^23 in the rounding direction wanted.  The three best are kept as
// floats that carry their index in the low bits.  One or two points within MARGIN of the best are then
// evaluated exactly by the thread; where three or more are that close, a warp evaluates all points and
// compares them in the order of its lanes.
// Bound: special-function unit (five operations a point, an eighth of the issue rate) beside the
// table's own bytes.  Measured for 1024 jobs x 71 pairs x 128 points (x 32 steps), all three outputs (43 MB):
// 134 us with a scan over s at every point and a launch of its own for the slabs, 44 us so.
constexpr int IDX_BITS = 7;               // points a thread can tell apart
constexpr int MAX_PARTS = 8;
constexpr int MAX_POINTS = MAX_PARTS << IDX_BITS;   // longer lists are evaluated exactly, all points
// Largest screening error (lg2.approx: 2^-22 |lg2 T| per operand, for times as extreme as 2^+-126) twice,
// and the index bits twice.
constexpr float MARGIN = 1e-4f;
// Quotients of whole numbers below this are at least 9.5e-7 away from the next integer (relative) or
// equal to it, so that a product with reciprocals, biased by 4e-7 towards the integer, rounds to the
// exact ceiling or floor.  Larger batch sizes are evaluated exactly, all points.
constexpr float EXACT_QUOTIENT = 1048576.f;
constexpr float LOW = 1.f - 4e-7f, HIGH = 1.f + 4e-7f;
constexpr float MAGIC = 12582912.f;

__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }

// per point of the grid, what does not depend on (K, class)
struct PointTable {
  float *m, *tg, *gl, *w, *qlo, *qhi;     // m; T_grad; gamma lg2 T_grad; phi / (T_grad m); M0 / m and Mmax / m, biased
};

// Goodput of two grid points at a (K, class), approximately; 0 where no s is feasible.
__device__ __forceinline__ float2 screen_two(float2 m, float2 tg, float2 gl, float2 w, float2 qlo, float2 qhi, float Kf,
                                             float rK, float ts, float gls, float rinv, float c0, float ig, float gs) {
  float2 ta = make_float2(0.f, 0.f);
  if (ts > 0.f) {
    const float2 d = __fadd2_rn(gl, f2(-gls));
    float2 e = make_float2(1.f + ex2_approx(-fabsf(d.x)), 1.f + ex2_approx(-fabsf(d.y)));
    e = __fmul2_rn(make_float2(lg2_approx(e.x), lg2_approx(e.y)), f2(ig));
    const float2 hi = make_float2(fmaxf(tg.x, ts), fmaxf(tg.y, ts));
    ta = __ffma2_rn(hi, make_float2(ex2_approx(e.x), ex2_approx(e.y)), __fmul2_rn(tg, f2(-1.f)));
  }
  const float2 km = __fmul2_rn(m, f2(Kf)), kr = __fmul2_rn(km, f2(rinv));
  const float2 ulo_ = __fadd2_rn(__ffma2_ru(qlo, f2(rK), f2(MAGIC)), f2(-MAGIC));
  const float2 uhi_ = __fadd2_rn(__ffma2_rd(qhi, f2(rK), f2(MAGIC)), f2(-MAGIC));
  const float2 ulo = make_float2(fmaxf(ulo_.x, 1.f), fmaxf(ulo_.y, 1.f)), uhi = make_float2(fminf(uhi_.x, gs), fminf(uhi_.y, gs));
  const float2 sq = __fmul2_rn(ta, __fmul2_rn(w, f2(rK)));
  float2 uc = make_float2(fminf(fmaxf(sqrt_approx(sq.x), ulo.x), uhi.x), fminf(fmaxf(sqrt_approx(sq.y), ulo.y), uhi.y));
  const float2 ua = __fadd2_rn(__fadd2_rd(uc, f2(MAGIC)), f2(-MAGIC));
  const float2 ub_ = __fadd2_rn(ua, f2(1.f));
  const float2 ub = make_float2(fminf(ub_.x, uhi.x), fminf(ub_.y, uhi.y));
  const float2 da = __fmul2_rn(__ffma2_rn(ua, tg, ta), __ffma2_rn(ua, kr, f2(c0)));
  const float2 db = __fmul2_rn(__ffma2_rn(ub, tg, ta), __ffma2_rn(ub, kr, f2(c0)));
  const float2 l = __fmul2_rn(ua, db), r = __fmul2_rn(ub, da);
  const float2 den = make_float2(l.x >= r.x ? da.x : db.x, l.y >= r.y ? da.y : db.y);
  const float2 num = __fmul2_rn(km, make_float2(l.x >= r.x ? ua.x : ub.x, l.y >= r.y ? ua.y : ub.y));
  float2 g = __fmul2_rn(num, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
  g.x = ulo.x <= uhi.x ? g.x : 0.f;
  g.y = ulo.y <= uhi.y ? g.y : 0.f;
  return g;
}

// The same of one sampled total batch size M (below 2^20; 0: none).  With many replicas neighbouring
// samples round to the same batch (m, s); `last` holds the batch of the sample before, and a sample that
// repeats it counts as none (of equal ones the smallest index is tabulated).
__device__ __forceinline__ float screen_sample(const JobModel &jm, float M, float Kf, float rK, float rmm, float ts,
                                               float gls, float rinv, float c0, float2 &last) {
  const float per_gpu = __fmaf_ru(M, rK * LOW, MAGIC) - MAGIC;
  const float u = __fmaf_ru(per_gpu, rmm * LOW, MAGIC) - MAGIC;           // s + 1
  const float m = __fmaf_ru(per_gpu, rcp_approx(u) * LOW, MAGIC) - MAGIC;
  const float run = Kf * m * u;
  const float tg = fmaf(jm.b_g, m, jm.a_g);
  float T = tg;
  if (ts > 0.f) {
    const float x = ex2_approx(-fabsf(jm.gamma * lg2_approx(tg) - gls));
    T = fmaxf(tg, ts) * ex2_approx(lg2_approx(1.f + x) * jm.inv_gamma);
  }
  const float g = run * rcp_approx(fmaf(u - 1.f, tg, T) * fmaf(run, rinv, c0));
  const bool use = M >= 1.f && run >= jm.M0 && run <= jm.Mmax && !(m == last.x && u == last.y);
  last = make_float2(m, u);
  return use ? g : 0.f;
}

// one goodput into the three best of a thread, carrying its index
__device__ __forceinline__ void keep_best(int &b1, int &b2, int &b3, float g, int idx) {
  int x = (__float_as_int(g) & ~((1 << IDX_BITS) - 1)) | idx;    // positive floats order as integers
  int y = min(b1, x);
  b1 = max(b1, x);
  x = min(b2, y);
  b2 = max(b2, y);
  b3 = max(b3, x);
}

template <bool SAMPLES>
__global__ void __maxnreg__(56) table_kernel(TableArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cl = cg::this_cluster();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");     // (who starts beside this waits for its end)
  const int KD = a.k_max + 1, tid = threadIdx.x, nthreads = blockDim.x;
  const int nb = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int j = a.j_first + (int)blockIdx.x / nb;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthreads >> 5;
  const TableLayout L = table_layout(KD, a.points, nthreads, (a.pair_count + nb - 1) / nb);
  const TableSmem t = {(float *)(smem + L.g), (uint16_t *)(smem + L.a)};
  int *s_best = (int *)(smem + L.best), *s_multi = (int *)(smem + L.multi);
  PointTable pt;
  pt.m = (float *)(smem + L.point);
  pt.tg = pt.m + a.points; pt.gl = pt.tg + a.points; pt.w = pt.gl + a.points; pt.qlo = pt.w + a.points; pt.qhi = pt.qlo + a.points;
  __shared__ int s_nmulti, s_nitem;
  if (tid == 0) { s_nmulti = 0; s_nitem = 0; }
  for (int i = tid; i < KD * 3; i += nthreads) { t.g[i] = 0.f; t.a[i] = 0xFFFFu; }
  __shared__ JobModel jm;
  if (tid == 0) jm = job_model(a.jp, j);
  __syncthreads();
  const int32_t *grid = a.m_grid + (size_t)j * a.G;
  const bool adapt = !SAMPLES || !a.adaptive || a.adaptive[j];
  const int mmax = SAMPLES ? a.m_max_gpu[j] : 1;
  const int G = !SAMPLES ? a.G : mmax < 1 ? 0 : adapt ? a.G : 1;
  const float rinv = adapt ? 1.f / (jm.phi + jm.M0) : 0.f;   // (phi + M) rinv = 1 / EFFICIENCY; 1 when fixed
  const float c0 = adapt ? jm.phi * rinv : 1.f;
  const float gs = (float)a.Gs, rmm = __frcp_rn((float)mmax);

  // ---- the points, in equal stretches; a point that repeats the one before it is never the smallest
  // index of its goodput and is left out
  bool big = !(jm.M0 < EXACT_QUOTIENT && (SAMPLES || jm.Mmax < EXACT_QUOTIENT));
  for (int i = tid; i < a.points; i += nthreads) {
    int v = 0, before = -1;
    if (i < G) {
      v = adapt ? grid[i] : (int)jm.M0;
      if (i > 0 && adapt) before = grid[i - 1];
    }
    const bool use = i < G && v != before && v >= 1;
    const float vf = (float)v;
    if (SAMPLES) {
      big |= use && !(vf < EXACT_QUOTIENT);
      pt.m[i] = use ? vf : 0.f;
    } else {
      const float tg = fmaf(jm.b_g, vf, jm.a_g), rm = __frcp_rn(vf);
      pt.m[i] = vf;
      pt.tg[i] = tg;
      pt.gl[i] = jm.gamma * lg2_approx(tg);
      pt.w[i] = __fdividef(jm.phi, tg * vf);
      pt.qlo[i] = use ? jm.M0 * rm * LOW : 1e6f * 1024.f;       // more steps than there are: not feasible
      pt.qhi[i] = use ? jm.Mmax * rm * HIGH : 0.f;
    }
  }
  const bool all_exact = __syncthreads_or(big) != 0 || a.points == 0;
  cl.sync();          // every block's results are cleared before any block publishes

  // this block's pairs: rank, rank + nb, ...
  const int mine = a.pair_count > rank ? (a.pair_count - rank + nb - 1) / nb : 0;
  auto pair_of = [&](int i) { return a.pairs[a.pair_first + rank + i * nb]; };
  auto exact = [&](float ts, int K, int i) {
    return SAMPLES ? sample_point(jm, ts, K, rinv, c0, mmax, adapt ? (long long)grid[i] : (long long)jm.M0, i)
                   : grid_point(jm, ts, (float)K, rinv, c0, grid[i], i, a.Gs);
  };
  auto tabulate = [&](int pr, const Best &b) {
    if (b.num > 0.f)
      publish(cl, t, (pr >> 2) * 3 + (pr & 3), b.num / b.den,
              (uint16_t)(SAMPLES ? b.tie : (b.tie & 0xFFFFu) * a.Gs + (b.tie >> 16)));
  };
  const int pb = nthreads / a.parts, part = tid / pb, ppp = a.points / a.parts;
  for (int first = 0; first < mine && !all_exact; first += pb) {
    const int pi = first + tid - part * pb;
    const bool on = part < a.parts && pi < mine;
    int b1 = 0, b2 = 0, b3 = 0, pr = 4;
    float ts = 0.f;
    if (on) {
      pr = pair_of(pi);
      const float Kf = (float)(pr >> 2), rK = __frcp_rn(Kf);
      ts = sync_time(jm, pr >> 2, pr & 3);
      const float gls = jm.gamma * lg2_approx(ts);
      const int at0 = part * ppp;
      float2 last = make_float2(0.f, 0.f);
      for (int k = 0; k < ppp; k += 4) {
        const int at = at0 + k;
        const float4 m = *(const float4 *)(pt.m + at);
        float g[4];
        if (SAMPLES) {
          g[0] = screen_sample(jm, m.x, Kf, rK, rmm, ts, gls, rinv, c0, last);
          g[1] = screen_sample(jm, m.y, Kf, rK, rmm, ts, gls, rinv, c0, last);
          g[2] = screen_sample(jm, m.z, Kf, rK, rmm, ts, gls, rinv, c0, last);
          g[3] = screen_sample(jm, m.w, Kf, rK, rmm, ts, gls, rinv, c0, last);
        } else {
          const float4 tg = *(const float4 *)(pt.tg + at), gl = *(const float4 *)(pt.gl + at), w = *(const float4 *)(pt.w + at),
                       qlo = *(const float4 *)(pt.qlo + at), qhi = *(const float4 *)(pt.qhi + at);
          const float2 x = screen_two(lo2(m), lo2(tg), lo2(gl), lo2(w), lo2(qlo), lo2(qhi), Kf, rK, ts, gls, rinv, c0, jm.inv_gamma, gs);
          const float2 y = screen_two(hi2(m), hi2(tg), hi2(gl), hi2(w), hi2(qlo), hi2(qhi), Kf, rK, ts, gls, rinv, c0, jm.inv_gamma, gs);
          g[0] = x.x; g[1] = x.y; g[2] = y.x; g[3] = y.y;
        }
#pragma unroll
        for (int z = 0; z < 4; ++z) keep_best(b1, b2, b3, g[z], k + z);
      }
    }
    if (first > 0) __syncthreads();        // the batch before has been read
    s_best[tid] = b1; s_best[nthreads + tid] = b2; s_best[2 * nthreads + tid] = b3;
    __syncthreads();
    int near = -1;         // first point << 12 | second point (0xFFF: none)
    if (tid < pb && on) {
      for (int p = 1; p < a.parts; ++p) b1 = max(b1, s_best[p * pb + tid]);
      if (b1 >= (1 << IDX_BITS)) {
        const int thr = __float_as_int(__int_as_float(b1 & ~((1 << IDX_BITS) - 1)) * (1.f - MARGIN));
        int n = 0, i0 = 0, i1 = 0;
        for (int p = 0; p < a.parts; ++p) {
#pragma unroll
          for (int z = 0; z < 3; ++z) {
            const int x = s_best[z * nthreads + p * pb + tid];
            if (x < thr) break;
            if (n == 0) i0 = p * ppp + (x & ((1 << IDX_BITS) - 1));
            else i1 = p * ppp + (x & ((1 << IDX_BITS) - 1));
            ++n;
          }
        }
        if (n >= 3) s_multi[atomicAdd(&s_nmulti, 1)] = pr;
        else near = (i0 << 12) | (n == 2 ? i1 : 0xFFF);
      }
    }
    // the first point by the pair's first thread, a second one by its second thread
    __syncthreads();
    if (tid < pb) s_best[tid] = near;
    __syncthreads();
    Best b = {0.f, 1.f, 0xFFFFFFFFu};
    if (on && part < 2) {
      near = s_best[tid - part * pb];
      const int i = part ? near & 0xFFF : near >> 12;
      if (near >= 0 && i != 0xFFF) {
        const Best o = exact(ts, pr >> 2, i);
        if (beats(o, b)) b = o;
      }
      if (part) { s_best[nthreads + tid] = __float_as_int(b.num); s_best[2 * nthreads + tid] = __float_as_int(b.den); s_best[tid] = (int)b.tie; }
    }
    __syncthreads();
    if (tid < pb && near >= 0) {
      if ((near & 0xFFF) != 0xFFF) {
        const Best o = {__int_as_float(s_best[nthreads + pb + tid]), __int_as_float(s_best[2 * nthreads + pb + tid]), (uint32_t)s_best[pb + tid]};
        if (beats(o, b)) b = o;
      }
      tabulate(pr, b);
    }
  }
  __syncthreads();
  // ---- pairs with several points that close (a job whose goodput hardly depends on m has dozens): a
  // warp finds the points again, a thread evaluates each, a warp compares a pair's points as they would
  // lie in its lanes (point i in lane i % 32).  The items take the place of s_best.
  int *s_item = s_best;                                             // [nthreads] place in s_multi << 16 | point
  float2 *s_value = (float2 *)(s_best + nthreads);                  // [nthreads] goodput as num / den
  uint32_t *s_span = (uint32_t *)s_multi + (a.pair_count + nb - 1) / nb;   // [pairs] first item << 16 | items
  const int nmulti = all_exact ? mine : s_nmulti;
  s_item[tid] = -1;                                   // (a pair that finds no room leaves its places empty)
  __syncthreads();
  for (int x = warp; x < nmulti; x += nwarps) {
    const int pr = all_exact ? pair_of(x) : s_multi[x], K = pr >> 2;
    const float ts = sync_time(jm, K, pr & 3);
    if (!all_exact && a.points <= 128) {
      // four points a lane: lane, lane + 32, ...
      const float Kf = (float)K, rK = __frcp_rn(Kf), gls = jm.gamma * lg2_approx(ts);
      float g[4];
#pragma unroll
      for (int q = 0; q < 4; q += 2) {
        const int i0 = min(lane + 32 * q, a.points - 1), i1 = min(lane + 32 * q + 32, a.points - 1);
        if (SAMPLES) {
          float2 last = make_float2(0.f, 0.f);
          g[q] = screen_sample(jm, pt.m[i0], Kf, rK, rmm, ts, gls, rinv, c0, last);
          last = make_float2(0.f, 0.f);
          g[q + 1] = screen_sample(jm, pt.m[i1], Kf, rK, rmm, ts, gls, rinv, c0, last);
        } else {
          auto two = [&](const float *v) { return make_float2(v[i0], v[i1]); };
          const float2 x = screen_two(two(pt.m), two(pt.tg), two(pt.gl), two(pt.w), two(pt.qlo), two(pt.qhi), Kf, rK, ts, gls, rinv,
                                      c0, jm.inv_gamma, gs);
          g[q] = x.x; g[q + 1] = x.y;
        }
        if (lane + 32 * q >= a.points) g[q] = 0.f;
        if (lane + 32 * q + 32 >= a.points) g[q + 1] = 0.f;
      }
      const float best = fmaxf(fmaxf(g[0], g[1]), fmaxf(g[2], g[3]));
      const float thr = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best))) * (1.f - MARGIN);
      unsigned bal[4];
      int found = 0, base = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) { bal[q] = __ballot_sync(0xffffffffu, g[q] >= thr); found += __popc(bal[q]); }
      if (lane == 0) base = atomicAdd(&s_nitem, found);
      base = __shfl_sync(0xffffffffu, base, 0);
      const bool room = base + found <= nthreads;
      if (lane == 0) s_span[x] = room ? ((uint32_t)base << 16) | (uint32_t)found : 0u;
      if (room) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if ((bal[q] >> lane) & 1u) s_item[base + __popc(bal[q] & ((1u << lane) - 1u))] = (x << 16) | (lane + 32 * q);
          base += __popc(bal[q]);
        }
        continue;
      }
    } else if (lane == 0 && !all_exact) {
      s_span[x] = 0u;
    }
    Best best = {0.f, 1.f, 0xFFFFFFFFu};              // all points (no room for items, or sizes beyond the screening)
    for (int i = lane; i < G; i += 32) {
      const Best p = exact(ts, K, i);
      if (beats(p, best)) best = p;
    }
    best = warp_best(best);
    if (lane == 0) tabulate(pr, best);
  }
  if (nmulti > 0 && !all_exact) {
    __syncthreads();
    uint32_t *s_tie = (uint32_t *)pt.m;               // [nthreads] (the screened points are done with; see table_layout)
    const int item = s_item[tid];
    if (item >= 0) {
      const int pr = s_multi[item >> 16];
      const Best b = exact(sync_time(jm, pr >> 2, pr & 3), pr >> 2, item & 0xFFFF);
      s_value[tid] = make_float2(b.num, b.den);
      s_tie[tid] = b.tie;
    }
    __syncthreads();
    for (int x = warp; x < nmulti; x += nwarps) {
      const int at = (int)(s_span[x] >> 16), n = (int)(s_span[x] & 0xFFFFu);
      if (n == 0) continue;
      Best best = {0.f, 1.f, 0xFFFFFFFFu};
      for (int q = 0; q < n; ++q) {
        const float2 v = s_value[at + q];
        const Best b = {v.x, v.y, s_tie[at + q]};
        if ((s_item[at + q] & 31) == lane && beats(b, best)) best = b;
      }
      best = warp_best(best);
      if (lane == 0) tabulate(s_multi[x], best);
    }
  }
  if (!a.speedup) {   // rack table alone: the local or node pair that holds the fair share is wanted too
    const int kf = a.fair_k[j], nf = a.fair_n[j];
    if (warp == 0 && kn_valid(kf, nf, a.k_max, a.n_max, a.kfit)) {
      const int cls = nf >= 2 ? CLS_NODE : CLS_LOCAL;
      const float ts = sync_time(jm, kf, cls);
      Best best = {0.f, 1.f, 0xFFFFFFFFu};
      for (int i = lane; i < G; i += 32) {
        const Best p = exact(ts, kf, i);
        if (beats(p, best)) best = p;
      }
      best = warp_best(best);
      if (lane == 0 && best.num > 0.f) t.g[kf * 3 + cls] = best.num / best.den;   // every block for itself
    }
  }
  cl.sync();          // all results are in every block's shared memory
  write_tables(a, t, (TableRow *)(smem + L.rows), j, rank, nb, fair_place(a, j));
}

// ---- small tables, long lists of points ------------------------------------------------------------
// Where there are few (job, K, class), evaluating every point by a warp each is a shorter chain than
// screening them: no table of points, no hand-over of the near ones, no blocks that wait for one another.
// Two launches then, the results per (K, class) in between in global memory; the second is launched beside the
// first (programmatic) and has its job's fair share ready when the results are there (0.6 us less than two launches
// one behind the other).  A warp's lanes evaluate the points lane, lane + 32, ..., MQ of them side by side.
template <bool SAMPLES, int MQ>
__global__ void __launch_bounds__(256, 4) sweep_kernel(TableArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int j = a.j_first + (int)blockIdx.x, lane = threadIdx.x & 31;
  const int x = (int)(blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5));
  int pr;
  if (x < a.pair_count) {
    pr = __ldg(a.pairs + a.pair_first + x);
  } else {            // (rack table alone: the pair that holds the fair share is wanted too)
    const int fair = x == a.pair_count && !a.speedup ? fair_place(a, j) : -1;
    if (fair < 0) return;
    pr = fair / 3 * 4 + fair % 3;
  }
  const JobModel jm = job_model(a.jp, j);
  const int32_t *grid = a.m_grid + (size_t)j * a.G;
  const bool adapt = !SAMPLES || !a.adaptive || a.adaptive[j];
  const int mmax = SAMPLES ? a.m_max_gpu[j] : 1;
  const int G = !SAMPLES ? a.G : mmax < 1 ? 0 : adapt ? a.G : 1;
  const float rinv = adapt ? 1.f / (jm.phi + jm.M0) : 0.f;   // (phi + M) rinv = 1 / EFFICIENCY; 1 when fixed
  const float c0 = adapt ? jm.phi * rinv : 1.f;
  const int K = pr >> 2;
  const float ts = sync_time(jm, K, pr & 3);
  Best best = {0.f, 1.f, 0xFFFFFFFFu};
  for (int i = lane; i < G; i += 32 * MQ) {
    if (SAMPLES) {
      const Best p = sample_point_inline(jm, ts, K, rinv, c0, mmax, adapt ? (long long)__ldg(grid + i) : (long long)jm.M0, i);
      if (beats(p, best)) best = p;
    } else {
      int m[MQ];
#pragma unroll
      for (int q = 0; q < MQ; ++q) m[q] = __ldg(grid + min(i + 32 * q, G - 1));
      grid_points<MQ>(jm, ts, (float)K, rinv, c0, m, i, (G - i + 31) / 32, a.Gs, a.one, a.zero, best);
    }
  }
  best = warp_best(best);
  if (lane == 0) {
    const size_t at = (size_t)j * (a.k_max + 1) * 3 + K * 3 + (pr & 3);
    const bool found = best.num > 0.f;
    a.g[at] = found ? best.num / best.den : 0.f;
    a.a[at] = !found ? (uint16_t)0xFFFFu : (uint16_t)(SAMPLES ? best.tie : (best.tie & 0xFFFFu) * a.Gs + (best.tie >> 16));
  }
}

__global__ void __launch_bounds__(256) slab_kernel(TableArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int KD = a.k_max + 1, j = a.j_first + (int)blockIdx.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");     // (who starts beside this waits for its end)
  const int fair = fair_place(a, j);
  const TableSmem t = {a.g + (size_t)j * KD * 3, a.a + (size_t)j * KD * 3};
  asm volatile("griddepcontrol.wait;" ::: "memory");
  write_tables(a, t, (TableRow *)smem, j, 0, 1, fair);
}

// REALLOC_FACTOR_j(delta) = (T_j - R_j delta) / (T_j + delta), clamped to [0, 1].
__global__ void realloc_factor_kernel(const float *__restrict__ age, const int32_t *__restrict__ restarts,
                                      float delta, int J, float *__restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  out[j] = realloc_factor(age[j], restarts[j], delta);
}

// Goodput-driven auto-scaling rule (Sec. 5.3): one thread per job.  All products are
// rounded one by one (no contraction): the comparisons decide integers.
__global__ void autoscale_kernel(const float *__restrict__ goodput, const int32_t *__restrict__ cur_nodes,
                                 int J, int k_max, int n_max, int gpn, float U, float L,
                                 int32_t *__restrict__ target_nodes) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  const int KD = k_max + 1, ND = n_max + 1;
  const float *g = goodput + (size_t)j * KD * ND;
  const float g1 = g[ND + 1];
  const int n = cur_nodes[j];
  const int limit = min(n_max, k_max / gpn);
  int target = n;
  if (n >= 1 && n <= limit && g1 > 0.f) {
    const float ideal_u = __fmul_rn(__fmul_rn(U, (float)(n * gpn)), g1);
    if (g[(size_t)(n * gpn) * ND + n] > ideal_u) {
      for (int t = n + 1; t <= limit; ++t) {
        const float ideal_l = __fmul_rn(__fmul_rn(L, (float)(t * gpn)), g1);
        if (g[(size_t)(t * gpn) * ND + t] >= ideal_l) target = t;
      }
    }
  }
  target_nodes[j] = target;
}

}  // namespace

int launch_autoscale(sched_ctx *ctx, const float *d_goodput, const int32_t *d_cur_nodes, int gpn, float U, float L,
                     int32_t *d_target_nodes) {
  const int J = ctx->cfg.num_jobs;
  if (J == 0) return SCHED_OK;
  autoscale_kernel<<<(J + 127) / 128, 128, 0, ctx->stream>>>(d_goodput, d_cur_nodes, J, ctx->cfg.k_max,
                                                             ctx->cfg.n_max, gpn, U, L, d_target_nodes);
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

// A block of at most eight warps per job and eight pairs; then one per job, an aligned four of the slab per
// thread (fewer than four warps make its first phase longer: 8 x 4, 64 jobs: 7.9 us with three, 6.6 so).
template <bool SAMPLES>
static int launch_small_table(sched_ctx *ctx, const TableArgs &a, int jobs) {
  const int warps = a.pair_count + (a.speedup ? 0 : 1);      // (the fair share's pair)
  if (warps > 0) {
    const int threads = 32 * std::min(8, warps);
    const dim3 grid((unsigned)jobs, (unsigned)((warps + 7) / 8));
    TimedLaunch tl_(ctx, KK_TABLE);
    if (SAMPLES || a.G <= 32) sweep_kernel<SAMPLES, 1><<<grid, threads, 0, ctx->stream>>>(a);
    else if (a.G <= 64) sweep_kernel<false, 2><<<grid, threads, 0, ctx->stream>>>(a);
    else sweep_kernel<false, 4><<<grid, threads, 0, ctx->stream>>>(a);
    SCHED_LAUNCH_CHECK(ctx);
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)jobs);
  lc.blockDim = dim3((unsigned)std::max(128, std::min(256, (ctx->KD * ctx->ND / 4 + 32) & ~31)));
  lc.dynamicSmemBytes = (size_t)(ctx->KD + 1) * sizeof(TableRow);
  lc.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = warps > 0 ? 1 : 0;
  {
    TimedLaunch tl_(ctx, KK_TABLE);
    SCHED_CUDA_CHECK(ctx, cudaLaunchKernelEx(&lc, slab_kernel, a));
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

// Whether the two launches above are the shorter way: the sweep's work (groups of 32 points, each with its
// steps) against the time of the one launch, which hardly depends on it up to 64 points, is a jump longer up to 128
// (several points come near one another) and far longer beyond (no room to note those: all points again).
// The lines lie where the two take the same time, measured for 2 x 2 to 128 x 8 GPUs and 8 to 1024 jobs (two
// launches / one, us): 4 x 4 GPUs with 32 points and 16 steps: 8 jobs 4.8 / 7.9, 384 jobs 8.5 / 8.9, 512 jobs 9.7 / 9.0;
// 16 x 4 with 64 points: 48 jobs 7.1 / 9.2, 96 jobs 10.5 / 9.5; 4 x 4 with 128 points: 256 jobs 12 / 14.5, 384
// jobs 14.1 / 16.0; 300 points, 4 x 4, 384 jobs: 29 / 46, 32 x 8, 256 jobs: 60 / 54; 300 samples, 16 x 4, 512 jobs: 77 / 106.
// (Contexts too large for any of this have no room for the results in between; a list too long for the screening
// takes this way wherever there is.)
static bool small_table(const sched_ctx *ctx, long long job_pairs, int G, int Gs, bool samples) {
  const long long work = job_pairs * ((G + 31) / 32) * (samples ? 32 : 32 + Gs);
  return ctx->d_gmax && (G > MAX_POINTS || work <= (G <= 64 ? 400000 : G <= 128 ? 1000000 : samples ? 20000000 : 8000000));
}

// A cluster of blocks per job: one block where the jobs alone give every SM two or where a job's (K, class)
// pairs fill no more than one, more otherwise, up to eight (large tables of few jobs gain as much as their
// sweep: each block writes its share of the slab).  A pair is shared by up to eight threads while all of
// them fit the GPU at once (registers: some 1170 threads per SM).  At least four warps, whatever the pairs
// are: pairs with several close points are spread over them (700 jobs x 11 pairs x 87 samples: 28.7 us
// with one warp and two threads per pair, 16.5 us).
template <bool SAMPLES>
static int launch_table(sched_ctx *ctx, TableArgs &a) {
  const int J = ctx->cfg.num_jobs;
  for (int j0 = 0; j0 < J; j0 += 65536) {
    const int jobs = std::min(65536, J - j0);
    a.j_first = j0;
    if (small_table(ctx, (long long)jobs * a.pair_count, a.G, a.Gs, SAMPLES)) {
      const int rc = launch_small_table<SAMPLES>(ctx, a, jobs);
      if (rc != SCHED_OK) return rc;
      continue;
    }
    int nb = 1;
    while (nb < 8 && jobs * nb < 2 * ctx->num_sms && a.pair_count * MAX_PARTS > 128 * nb) nb *= 2;
    const int pairs = std::max(1, (a.pair_count + nb - 1) / nb);
    // (at least two: the second evaluates a second point)
    int parts = MAX_PARTS;
    while (parts > 2 && (a.G < 4 * parts || pairs * parts > 512 ||
                         (long long)jobs * nb * pairs * parts > 1024LL * ctx->num_sms))
      parts /= 2;
    while (parts < MAX_PARTS && (a.G + parts - 1) / parts > (1 << IDX_BITS)) parts *= 2;
    const int ppp = (((a.G + parts - 1) / parts) + 3) & ~3;
    a.parts = parts;
    a.points = a.G <= MAX_POINTS ? ppp * parts : 0;
    const int threads = std::max(128, std::min(512, (pairs * parts + 31) & ~31));
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(jobs * nb));
    lc.blockDim = dim3((unsigned)threads);
    lc.dynamicSmemBytes = table_layout(ctx->KD, a.points, threads, pairs).total;
    lc.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)nb;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    if (lc.dynamicSmemBytes > 48 * 1024)
      SCHED_CUDA_CHECK(ctx, cudaFuncSetAttribute(table_kernel<SAMPLES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lc.dynamicSmemBytes));
    {
      TimedLaunch tl_(ctx, KK_TABLE);
      SCHED_CUDA_CHECK(ctx, cudaLaunchKernelEx(&lc, table_kernel<SAMPLES>, a));
    }
    SCHED_LAUNCH_CHECK(ctx);
  }
  return SCHED_OK;
}

static TableArgs table_args(const sched_ctx *ctx, const sched_jobs *jobs) {
  const sched_config &c = ctx->cfg;
  TableArgs a = {};
  a.jp = {jobs->alpha_grad, jobs->beta_grad, jobs->alpha_local, jobs->beta_local, jobs->alpha_node, jobs->beta_node,
          nullptr, nullptr, jobs->gamma, jobs->phi, jobs->m0, jobs->m_max_total};
  a.m_grid = jobs->m_grid;
  a.pairs = ctx->d_pairs;
  a.pair_count = ctx->num_pairs;
  a.g = ctx->d_gmax; a.a = ctx->d_amax;
  a.one = 1.f; a.zero = 0.f;
  a.kfit = ctx->d_kfit; a.nmin = ctx->d_nmin; a.fair_k = jobs->fair_k; a.fair_n = jobs->fair_n;
  a.k_max = c.k_max; a.n_max = c.n_max; a.G = c.grid_m; a.Gs = c.grid_s;
  return a;
}

// d_speedup_rack (with the rack pair) may be NULL; so may d_speedup: then only the table of the rack
// class is built (allocations whose nodes lie in two or more racks), over the same fair-share goodput.
int launch_speedup_table(sched_ctx *ctx, const sched_jobs *jobs, float *d_goodput, float *d_speedup, uint16_t *d_argmax,
                         const float *d_alpha_rack, const float *d_beta_rack, float *d_goodput_rack, float *d_speedup_rack,
                         uint16_t *d_argmax_rack) {
  if (ctx->cfg.num_jobs == 0) return SCHED_OK;
  TableArgs a = table_args(ctx, jobs);
  a.goodput = d_goodput; a.speedup = d_speedup; a.argmax = d_argmax;
  if (d_speedup_rack) {
    a.jp.alpha_rack = d_alpha_rack; a.jp.beta_rack = d_beta_rack;
    a.goodput_rack = d_goodput_rack; a.speedup_rack = d_speedup_rack; a.argmax_rack = d_argmax_rack;
    if (d_speedup) a.pair_count += ctx->num_rack_pairs;
    else { a.pair_first = ctx->num_pairs; a.pair_count = ctx->num_rack_pairs; }
  }
  return launch_table<false>(ctx, a);
}

int launch_speedup_table_msample(sched_ctx *ctx, const sched_jobs *jobs, const int32_t *d_m_samples, int G,
                                 const int32_t *d_m_max_gpu, const uint8_t *d_adaptive, float *d_goodput,
                                 float *d_speedup, uint16_t *d_argmax) {
  if (ctx->cfg.num_jobs == 0) return SCHED_OK;
  TableArgs a = table_args(ctx, jobs);
  a.m_grid = d_m_samples; a.m_max_gpu = d_m_max_gpu; a.adaptive = d_adaptive; a.G = G;
  a.goodput = d_goodput; a.speedup = d_speedup; a.argmax = d_argmax;
  return launch_table<true>(ctx, a);
}

int launch_realloc_factor(sched_ctx *ctx, const sched_jobs *jobs, float *d_out) {
  const int J = ctx->cfg.num_jobs;
  if (J == 0) return SCHED_OK;
  {
  TimedLaunch tl_(ctx, KK_REALLOC);
  realloc_factor_kernel<<<(J + 127) / 128, 128, 0, ctx->stream>>>(jobs->age_sec, jobs->num_restarts,
                                                                   ctx->cfg.delta_sec, J, d_out);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}
