// Population-search operators (Sec. 4.3): ranking, parent selection + row-wise crossover
// + row perturbation, and the repair that enforces node capacity and interference
// avoidance (Sec. 4.2).  Integer work only; all randomness comes from the counter-based
// stream, so every output is a pure function of the inputs.
//
// Implementations of the same operators on dense matrices, chosen by shape:
//  * child_kernel: one launch, a block or a cluster of blocks per child, rows of any width up to 512 nodes (the
//    entry points called on their own, and dense rounds without summaries);
//  * rows2_kernel + colrepair_kernel: rows of whole 16-byte vectors and at most 512 nodes, with per-row summaries or
//    more jobs than child_kernel's counters hold - batched rows with fused column sums and occupant lists, a work list of
//    violating nodes;
//  * rows_kernel + cols_kernel (+ rank_kernel): the general pair - a warp per (candidate, job)
//    row through shared memory, then a thread per (candidate, node) column.
// Rounds do not use dense matrices for their generations (round_flow.cu, rowstore.cu) unless neither the
// blocks nor the memory of those fit.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "fitness_common.cuh"
#include "search_common.cuh"

namespace {

enum { ROWS_GENERATION = 0, ROWS_INIT = 1, ROWS_REPAIR = 2 };

// rank[i] = number of candidates ordered before i (fitness descending, index ascending)
__global__ void __launch_bounds__(128)
rank_kernel(const uint32_t *__restrict__ fitness_bits, int P, int32_t *__restrict__ rank,
            int32_t *__restrict__ order) {
  __shared__ uint32_t tile[128];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t ki = (i < P) ? order_key(fitness_bits[i]) : 0u;
  int r = 0;
  for (int base = 0; base < P; base += 128) {
    const int o = base + threadIdx.x;
    tile[threadIdx.x] = (o < P) ? order_key(fitness_bits[o]) : 0u;
    __syncthreads();
    const int lim = min(128, P - base);
    for (int t = 0; t < lim; ++t) {
      const uint32_t ko = tile[t];
      r += (ko > ki || (ko == ki && base + t < i)) ? 1 : 0;
    }
    __syncthreads();
  }
  if (i < P) {
    rank[i] = r;
    order[r] = i;
  }
}

struct RowsArgs {
  const int16_t *src;       // parents [P][J][N], or the current allocation [J][N] (may be NULL), or dst
  int16_t *dst;             // children [count][J][N]
  const int16_t *cap;       // [N]
  const int32_t *k_cap;     // [J] or NULL
  const uint8_t *active;    // [J] or NULL
  const int32_t *rank;      // [P]   (generation mode)
  const int32_t *order;     // [P]
  const uint32_t *fitness_bits;  // [P] parents' fitness (generation mode)
  uint8_t *dflag;           // [count][J]
  const int16_t *cur;       // [J][N] current allocation for the summaries' "changed" bit, or NULL
  uint32_t *summ;           // [count][J] row summaries (batched kernels only), or NULL
  const uint32_t *summ_in;  // [P][J] summaries of the parents (generation mode), or NULL
  int mode, P, J, num_nodes, k_max, n_max, num_elite, count;
  uint32_t thr, gen, first_cand;
  RngKey key;
};

__global__ void __launch_bounds__(256) rows_kernel(RowsArgs a) {
  extern __shared__ __align__(16) int16_t s_rows[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long gw = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
  if (gw >= (long long)a.count * a.J) return;
  const int cl = (int)(gw / a.J), j = (int)(gw % a.J);
  const uint32_t c = a.first_cand + (uint32_t)cl;
  const int NN = a.num_nodes;
  const int row_stride = (NN + 7) & ~7;
  int16_t *row = s_rows + (size_t)warp * row_stride;
  int16_t *out = a.dst + ((size_t)cl * a.J + j) * NN;
  const bool vec = ((NN & 7) == 0) && ((((uintptr_t)a.dst | (uintptr_t)a.src) & 15) == 0);

  if (a.active && !a.active[j]) {
    if (vec) for (int v = lane; v < NN / 8; v += 32) ((uint4 *)out)[v] = make_uint4(0, 0, 0, 0);
    else for (int n = lane; n < NN; n += 32) out[n] = 0;
    if (lane == 0) a.dflag[(size_t)cl * a.J + j] = 0;
    return;
  }

  // which row feeds this child row, and the perturbation draw
  const int16_t *src = nullptr;
  bool mutate = false;
  u32x4 mw = {0, 0, 0, 0};
  if (a.mode == ROWS_GENERATION) {
    int parent;
    if ((int)c < a.num_elite) {
      parent = a.order[c];
    } else {
      const u32x4 s = draw(a.key, 0u, c, a.gen, SLOT_SELECT);
      const int i0 = bounded(s.x, a.P), i1 = bounded(s.y, a.P);
      const int i2 = bounded(s.z, a.P), i3 = bounded(s.w, a.P);
      const int pa = a.rank[i0] <= a.rank[i1] ? i0 : i1;
      const int pb = a.rank[i2] <= a.rank[i3] ? i2 : i3;
      const u32x4 x = draw(a.key, (uint32_t)j, c, a.gen, SLOT_XOVER);
      parent = (x.x >> 31) ? pb : pa;
      mw = draw(a.key, (uint32_t)j, c, a.gen, SLOT_MUTATE);
      mutate = mw.x < a.thr;
    }
    src = a.src + ((size_t)parent * a.J + j) * NN;
  } else if (a.mode == ROWS_INIT) {
    src = a.src ? a.src + (size_t)j * NN : nullptr;
    if (c > 0) {
      mw = draw(a.key, (uint32_t)j, c, GEN_INIT, SLOT_INIT);
      mutate = mw.x < a.thr;
    }
  } else {
    src = out;
  }

  // load into shared memory, every entry forced into [0, capacity of its node]
  int K = 0, N = 0;
  if (!src) {
    for (int n = lane; n < row_stride; n += 32) row[n] = 0;
  } else if (vec) {
    for (int v = lane; v < NN / 8; v += 32) {
      uint4 x = __ldg((const uint4 *)src + v);
      const uint4 cp = __ldg((const uint4 *)a.cap + v);
      x.x = __vimin_s16x2_relu(x.x, __vimax_s16x2_relu(cp.x, 0u));
      x.y = __vimin_s16x2_relu(x.y, __vimax_s16x2_relu(cp.y, 0u));
      x.z = __vimin_s16x2_relu(x.z, __vimax_s16x2_relu(cp.z, 0u));
      x.w = __vimin_s16x2_relu(x.w, __vimax_s16x2_relu(cp.w, 0u));
      ((uint4 *)row)[v] = x;
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        K += (int)(w[q] & 0xFFFFu) + (int)(w[q] >> 16);
        N += ((w[q] & 0xFFFFu) != 0u) + ((w[q] >> 16) != 0u);
      }
    }
  } else {
    for (int n = lane; n < NN; n += 32) {
      const int cp = max((int)a.cap[n], 0);
      const int v = min(max((int)src[n], 0), cp);
      row[n] = (int16_t)v;
      K += v;
      N += v > 0;
    }
  }
  K = warp_sum(K);
  N = warp_sum(N);
  __syncwarp();

  if (mutate) {
    const uint32_t op = bounded(mw.y, 3u);
    if (op == 0u) {
      const int n = (int)bounded(mw.w, (uint32_t)NN);
      if (lane == 0) row[n] = (int16_t)min((int)row[n] + 1, max((int)a.cap[n], 0));
    } else if (N > 0) {
      const int ns = nth_occupied(row, NN, bounded(mw.z, (uint32_t)N), lane);
      if (op == 1u) {
        if (lane == 0) row[ns] = (int16_t)(row[ns] - 1);
      } else {
        const int nd = (int)bounded(mw.w, (uint32_t)NN);
        if (nd != ns && lane == 0) {
          row[nd] = (int16_t)min((int)row[nd] + (int)row[ns], max((int)a.cap[nd], 0));
          row[ns] = 0;
        }
      }
    }
    __syncwarp();
    K = 0; N = 0;
    for (int n = lane; n < NN; n += 32) { K += row[n]; N += row[n] > 0; }
    K = warp_sum(K);
    N = warp_sum(N);
  }

  // per-row caps: replicas above the job's cap leave from the highest node index down,
  // then occupied nodes beyond n_max are cleared from the highest index down
  int kc = a.k_cap ? a.k_cap[j] : a.k_max;
  kc = max(0, min(kc, a.k_max));
  if (K > kc || N > a.n_max) {
    if (lane == 0) {
      int excess = K - kc;
      for (int n = NN - 1; n >= 0 && excess > 0; --n) {
        const int take = min((int)row[n], excess);
        row[n] = (int16_t)(row[n] - take);
        excess -= take;
      }
      int occ = 0;
      for (int n = 0; n < NN; ++n) {
        if (row[n] > 0) {
          ++occ;
          if (occ > a.n_max) row[n] = 0;
        }
      }
      N = min(occ, a.n_max);
    }
    N = __shfl_sync(0xffffffffu, N, 0);
    __syncwarp();
  }

  if (vec) for (int v = lane; v < NN / 8; v += 32) ((uint4 *)out)[v] = ((const uint4 *)row)[v];
  else for (int n = lane; n < NN; n += 32) out[n] = row[n];
  if (lane == 0) a.dflag[(size_t)cl * a.J + j] = (N >= 2) ? 1 : 0;
}

struct ColsArgs {
  int16_t *pop;             // [count][J][N], repaired in place
  const uint8_t *dflag;     // [count][J]
  const int16_t *cap;
  int J, num_nodes, count;
  uint32_t gen, first_cand;
  RngKey key;
};

// One thread per (candidate, node).  Interference avoidance: of the jobs flagged as
// distributed that occupy the node, only the first in job order rotated by the node's
// draw stays.  Capacity: GPUs above the node's size are taken from its jobs in job order
// rotated by a second draw.
__global__ void __launch_bounds__(128) cols_kernel(ColsArgs a) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int cl = blockIdx.y;
  if (n >= a.num_nodes) return;
  const uint32_t c = a.first_cand + (uint32_t)cl;
  const int J = a.J, NN = a.num_nodes;
  int16_t *col = a.pop + (size_t)cl * J * NN + n;
  const uint8_t *df = a.dflag + (size_t)cl * J;
  int total = 0, nelig = 0;
#pragma unroll 8
  for (int j = 0; j < J; ++j) {
    const int v = col[(size_t)j * NN];
    total += v;
    nelig += (v > 0 && df[j]) ? 1 : 0;
  }
  const int cp = max((int)a.cap[n], 0);
  if (nelig <= 1 && total <= cp) return;
  if (nelig >= 2) {
    const int o = (int)bounded(draw(a.key, (uint32_t)n, c, a.gen, SLOT_REPAIR_INTF).x, (uint32_t)J);
    int keep = -1, best = J;
    for (int j = 0; j < J; ++j) {
      if (df[j] && col[(size_t)j * NN] > 0) {
        int t = j - o;
        if (t < 0) t += J;
        if (t < best) { best = t; keep = j; }
      }
    }
    for (int j = 0; j < J; ++j) {
      if (j != keep && df[j]) {
        const int v = col[(size_t)j * NN];
        if (v > 0) { total -= v; col[(size_t)j * NN] = 0; }
      }
    }
  }
  int excess = total - cp;
  if (excess > 0) {
    const int o = (int)bounded(draw(a.key, (uint32_t)n, c, a.gen, SLOT_REPAIR_CAP).x, (uint32_t)J);
    for (int t = 0; t < J && excess > 0; ++t) {
      int j = o + t;
      if (j >= J) j -= J;
      const int v = col[(size_t)j * NN];
      if (v > 0) {
        const int take = min(v, excess);
        col[(size_t)j * NN] = (int16_t)(v - take);
        excess -= take;
      }
    }
  }
}

// index of the best candidate (largest key, lowest index on ties) and its fitness
__global__ void __launch_bounds__(256)
best_index_kernel(const uint32_t *__restrict__ fitness_bits, int P, int32_t *__restrict__ best_idx,
                  float *__restrict__ best_fitness) {
  __shared__ unsigned long long s[256];
  unsigned long long best = 0ull;   // (key << 32) | (0xFFFFFFFF - index): larger is better
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    const unsigned long long v = ((unsigned long long)order_key(fitness_bits[i]) << 32) |
                                 (unsigned long long)(0xFFFFFFFFu - (uint32_t)i);
    best = v > best ? v : best;
  }
  s[threadIdx.x] = best;
  __syncthreads();
  for (int off = 128; off >= 1; off >>= 1) {
    if ((int)threadIdx.x < off) s[threadIdx.x] = s[threadIdx.x] > s[threadIdx.x + off] ? s[threadIdx.x] : s[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int idx = (int)(0xFFFFFFFFu - (uint32_t)(s[0] & 0xFFFFFFFFull));
    *best_idx = idx;
    if (best_fitness) *best_fitness = __uint_as_float(fitness_bits[idx]);
  }
}

__global__ void copy_best_kernel(const int16_t *__restrict__ pop, const int32_t *__restrict__ best_idx,
                                 size_t elems, int16_t *__restrict__ out) {
  const int16_t *src = pop + (size_t)(*best_idx) * elems;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = src[i];
}


// ---------------------------------------------------------------------------------------
// Batched row kernel with fused column sums (rows of at most 64 16-byte vectors).
//
// A block owns 256 consecutive rows of one candidate, a warp 32 of them.  Each lane draws
// the crossover / perturbation words of "its" row once (32 Philox calls run side by side
// instead of one per warp), then the warp walks the 32 rows: one 16-byte load per lane and
// vector, clamp, row totals by shuffle, store.  Rows that are perturbed or break a row cap
// detour through shared memory.  While walking, every lane accumulates, for its own
// columns, the GPUs placed and the number of distributed jobs; the block's column partials
// go to scratch, so the column pass never re-reads the population.
// ---------------------------------------------------------------------------------------
// Occupants of a node recorded per (candidate, row batch, node); a node with more occupants in
// one batch than this falls back to scanning the column.
constexpr int OCC_SLOTS = 8;

struct Rows2Args {
  RowsArgs r;
  int32_t *colsum;   // [count][nbatch][num_nodes] GPUs placed on the node by the batch's rows
  int32_t *colelig;  // same shape: rows of the batch that are distributed and occupy the node
  unsigned int *list_count;  // length of the column work list (zeroed before this kernel)
  uint32_t *list;            // the work list: (candidate << 13 | node) of nodes that need repair
  unsigned int *cand_ticket; // [count] blocks of the candidate that have finished (self-resetting)
  int32_t *occ_count;        // [count][nbatch][num_nodes] rows of the batch that occupy the node
  uint32_t *occ_list;        // [count][nbatch][num_nodes][OCC_SLOTS] job | GPUs << 20 | distributed << 31
  int nbatch, lpr_log2;
};

__device__ __forceinline__ uint4 clamp_vec(uint4 x, uint4 cp) {
  x.x = __vimin_s16x2_relu(x.x, cp.x);
  x.y = __vimin_s16x2_relu(x.y, cp.y);
  x.z = __vimin_s16x2_relu(x.z, cp.z);
  x.w = __vimin_s16x2_relu(x.w, cp.w);
  return x;
}

// K in the low 22 bits, occupied-node count in the high 10 (entries are >= 0 here)
__device__ __forceinline__ uint32_t row_partial(uint4 x) {
  int k = __dp2a_lo((int)x.x, 0x0101, 0);
  k = __dp2a_lo((int)x.y, 0x0101, k);
  k = __dp2a_lo((int)x.z, 0x0101, k);
  k = __dp2a_lo((int)x.w, 0x0101, k);
  const uint32_t o = __vimin_s16x2_relu(x.x, 0x00010001u) + __vimin_s16x2_relu(x.y, 0x00010001u) +
                     __vimin_s16x2_relu(x.z, 0x00010001u) + __vimin_s16x2_relu(x.w, 0x00010001u);
  return (uint32_t)k | (((o & 0xFFFFu) + (o >> 16)) << 22);
}

struct ColfixArgs {
  int16_t *pop;
  const uint8_t *dflag;
  const int16_t *cap;
  const int32_t *colsum, *colelig;
  uint32_t *summ;           // [count][J] row summaries to keep in step with the removals, or NULL
  const int16_t *cur;       // current allocation (for the summaries' differing-entries count), or NULL
  const int32_t *occ_count; // per (candidate, row batch, node) occupants recorded by the row kernel
  const uint32_t *occ_list;
  uint32_t *list;           // work list of (candidate << 13 | node) entries
  unsigned int *list_count;
  int J, num_nodes, nbatch;
  uint32_t gen, first_cand;
  RngKey key;
};

// A column-pass write A[j][n]: v_old -> v_new keeps row j's summary in step:
// K += v_new - v_old, N -= 1 if the entry became empty, and the count of entries that
// differ from the current allocation is adjusted.  The three fields never leave their
// ranges, so one wrapped 32-bit add does all three.
__device__ __forceinline__ void summ_update(const ColfixArgs &a, uint32_t *summ_c, int j, int n, int v_old, int v_new) {
  if (!summ_c) return;
  int d_diff = 0;
  if (a.cur) {
    const int cv = a.cur[(size_t)j * a.num_nodes + n];
    d_diff = (int)(v_new != cv) - (int)(v_old != cv);
  }
  const uint32_t delta = (uint32_t)(v_new - v_old) + ((uint32_t)((v_new == 0 && v_old > 0) ? -1 : 0) << 11) +
                         ((uint32_t)d_diff << 22);
  atomicAdd(summ_c + j, delta);
}

// Repair of one column by a whole warp (any J): interference, then capacity, each with a
// few passes over the column; loads are issued in batches so that they overlap.
__device__ __noinline__ void repair_column_any(const ColfixArgs &a, uint32_t *summ_c, int cl, int nn, int tot, int ne,
                                               int cap_n, int lane) {
  const uint32_t c = a.first_cand + (uint32_t)cl;
  const int J = a.J, NN = a.num_nodes;
  const uint8_t *df = a.dflag + (size_t)cl * J;
  {
    int16_t *col = a.pop + (size_t)cl * J * NN + nn;
    // the loops below first issue a batch of independent column loads, then work on them
    constexpr int U = 8;
    if (ne >= 2) {
      const int o = (int)bounded(draw(a.key, (uint32_t)nn, c, a.gen, SLOT_REPAIR_INTF).x, (uint32_t)J);
      int best = J;
      for (int jb = 0; jb < J; jb += 32 * U) {
        int v[U], d[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int j = jb + 32 * k + lane;
          v[k] = (j < J) ? (int)col[(size_t)j * NN] : 0;
          d[k] = (j < J) ? (int)df[j] : 0;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
          if (d[k] && v[k] > 0) {
            int t = jb + 32 * k + lane - o;
            if (t < 0) t += J;
            best = min(best, t);
          }
        }
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, off));
      int keep = o + best;
      if (keep >= J) keep -= J;
      int removed = 0;
      for (int jb = 0; jb < J; jb += 32 * U) {
        int v[U], d[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int j = jb + 32 * k + lane;
          v[k] = (j < J) ? (int)col[(size_t)j * NN] : 0;
          d[k] = (j < J) ? (int)df[j] : 0;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int j = jb + 32 * k + lane;
          if (d[k] && v[k] > 0 && j != keep) {
            col[(size_t)j * NN] = 0;
            removed += v[k];
            summ_update(a, summ_c, j, nn, v[k], 0);
          }
        }
      }
      tot -= warp_sum(removed);
    }
    int excess = tot - cap_n;
    if (excess > 0) {
      const int o = (int)bounded(draw(a.key, (uint32_t)nn, c, a.gen, SLOT_REPAIR_CAP).x, (uint32_t)J);
      constexpr int C = 4;   // chunks of 32 jobs loaded together
      for (int t0 = 0; t0 < J && excess > 0; t0 += 32 * C) {
        int v[C], jj[C];
#pragma unroll
        for (int k = 0; k < C; ++k) {
          const int t = t0 + 32 * k + lane;
          int j = o + t;
          if (j >= J) j -= J;
          jj[k] = j;
          v[k] = (t < J) ? (int)col[(size_t)j * NN] : 0;
        }
#pragma unroll
        for (int k = 0; k < C; ++k) {
          if (excess <= 0) break;
          int s = v[k];                                // inclusive prefix over the 32 jobs
#pragma unroll
          for (int off = 1; off < 32; off <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, s, off);
            if (lane >= off) s += u;
          }
          const int take = min(v[k], max(excess - (s - v[k]), 0));
          if (take > 0) {
            col[(size_t)jj[k] * NN] = (int16_t)(v[k] - take);
            summ_update(a, summ_c, jj[k], nn, v[k], v[k] - take);
          }
          excess -= __shfl_sync(0xffffffffu, s, 31);
        }
      }
    }
  }
}

// Repair of one column from its occupants, one occupant per lane (entry = job | GPUs << 20 |
// distributed << 31 in the first have_n lanes): no pass over the column.
__device__ void repair_column_entries(const ColfixArgs &a, uint32_t *summ_c, int cl, int nn, int tot, int ne,
                                      int cap_n, int lane, uint32_t entry, int have_n) {
  const uint32_t c = a.first_cand + (uint32_t)cl;
  const int J = a.J, NN = a.num_nodes;
  const bool have = lane < have_n;
  const int j = (int)(entry & 0xFFFFFu);
  int v = have ? (int)((entry >> 20) & 0x7FFu) : 0;
  const bool dist = have && (entry >> 31);
  int16_t *col = a.pop + (size_t)cl * J * NN + nn;
  if (ne >= 2) {
    const int o = (int)bounded(draw(a.key, (uint32_t)nn, c, a.gen, SLOT_REPAIR_INTF).x, (uint32_t)J);
    int t = J;
    if (dist && v > 0) { t = j - o; if (t < 0) t += J; }
    int best = t;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, off));
    int removed = 0;
    if (dist && v > 0 && t != best) {
      col[(size_t)j * NN] = 0;
      summ_update(a, summ_c, j, nn, v, 0);
      removed = v;
      v = 0;
    }
    tot -= warp_sum(removed);
  }
  const int excess = tot - cap_n;
  if (excess > 0) {
    const int o = (int)bounded(draw(a.key, (uint32_t)nn, c, a.gen, SLOT_REPAIR_CAP).x, (uint32_t)J);
    int rot = 0x7fffffff;
    if (have) { rot = j - o; if (rot < 0) rot += J; }
    int ahead = 0;                       // GPUs of the occupants that come first in rotated order
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const int rk = __shfl_sync(0xffffffffu, rot, k);
      const int vk = __shfl_sync(0xffffffffu, v, k);
      if (rk < rot) ahead += vk;
    }
    const int take = have ? min(v, max(excess - ahead, 0)) : 0;
    if (take > 0) {
      col[(size_t)j * NN] = (int16_t)(v - take);
      summ_update(a, summ_c, j, nn, v, v - take);
    }
  }
}

// Occupants gathered from the per-batch lists the row kernel left in global memory.  Falls
// back to the column scan when a batch overflowed its slots or the node has more than 32
// occupants.
__device__ void repair_column_list(const ColfixArgs &a, int cl, int nn, int tot, int ne, int cap_n, int lane) {
  const int NN = a.num_nodes;
  uint32_t *summ_c = a.summ ? a.summ + (size_t)cl * a.J : nullptr;
  uint32_t entry = 0;
  int have_n = 0;
  bool overflow = false;
  for (int b = 0; b < a.nbatch; ++b) {
    const size_t at = ((size_t)cl * a.nbatch + b) * NN + nn;
    const int cb = a.occ_count[at];
    overflow |= cb > OCC_SLOTS;
    const int take_n = min(cb, OCC_SLOTS);
    if (lane >= have_n && lane < have_n + take_n) entry = a.occ_list[at * OCC_SLOTS + (lane - have_n)];
    have_n += take_n;
  }
  if (overflow || have_n > 32) repair_column_any(a, summ_c, cl, nn, tot, ne, cap_n, lane);
  else repair_column_entries(a, summ_c, cl, nn, tot, ne, cap_n, lane, entry, have_n);
}

// VPL = 16-byte vectors per lane; a row is split over LPR = 1 << LPR_LOG2 lanes
// (LPR * VPL >= row_vecs, FULL when equal), so a warp works on 32 / LPR rows at a time.
template <int LPR_LOG2, int VPL, bool FULL>
__global__ void __launch_bounds__(256, 4) rows2_kernel(Rows2Args aa) {
  const RowsArgs &a = aa.r;
  constexpr int MAXN = 8 * (1 << LPR_LOG2) * VPL;   // nodes this instantiation can hold
  constexpr int QCAP = 64;                          // vectors in a warp's occupant queue
  __shared__ __align__(16) int16_t s_row[8][MAXN];  // per-warp detour buffer
  __shared__ __align__(16) int16_t s_cap[MAXN];     // node sizes floored at 0
  __shared__ int32_t s_tot[MAXN], s_el[MAXN], s_cnt[MAXN];
  __shared__ uint32_t s_occ[MAXN * OCC_SLOTS];
  __shared__ int s_parent[2];
  // per-warp queue of non-empty vectors waiting to be expanded into occupants
  __shared__ __align__(16) uint4 s_qvec[8][QCAP];
  __shared__ uint32_t s_qmeta[8][QCAP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cl = blockIdx.y, batch = blockIdx.x;
  const uint32_t c = a.first_cand + (uint32_t)cl;
  const int NN = a.num_nodes, J = a.J;
  const int row_vecs = NN >> 3;
  constexpr int LPR = 1 << LPR_LOG2, RPI = 32 >> LPR_LOG2;        // lanes per row, rows per iteration
  const int grp = lane >> LPR_LOG2, sub = lane & (LPR - 1);
  const unsigned gmask = (LPR == 32) ? 0xffffffffu : (((1u << LPR) - 1u) << (grp * LPR));
  for (int i = threadIdx.x; i < NN; i += blockDim.x) {
    s_tot[i] = 0; s_el[i] = 0; s_cnt[i] = 0;
    s_cap[i] = (int16_t)max((int)a.cap[i], 0);
  }

  // ---- parents of this candidate (generation mode), found by the block itself -------------
  // rank(i) = number of candidates ordered before i (fitness descending, index ascending).
  // An elite child needs the candidate of rank c; any other child the better-ranked of two
  // random pairs, which the two candidates' own keys and indices decide.
  if (a.mode == ROWS_GENERATION) {
    const int P = a.P;
    if ((int)c < a.num_elite) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const uint32_t ki = order_key(a.fitness_bits[i]);
        int rk = 0;
        for (int o = 0; o < P; ++o) {
          const uint32_t ko = order_key(__ldg(a.fitness_bits + o));
          rk += (ko > ki || (ko == ki && o < i)) ? 1 : 0;
        }
        if (rk == (int)c) s_parent[0] = s_parent[1] = i;
      }
    } else {
      const u32x4 sel = draw(a.key, 0u, c, a.gen, SLOT_SELECT);
      const int idx[4] = {(int)bounded(sel.x, P), (int)bounded(sel.y, P), (int)bounded(sel.z, P),
                          (int)bounded(sel.w, P)};
      if (threadIdx.x == 0) {
        uint32_t k4[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) k4[q] = order_key(__ldg(a.fitness_bits + idx[q]));
        s_parent[0] = tournament_winner(k4[0], idx[0], k4[1], idx[1]);
        s_parent[1] = tournament_winner(k4[2], idx[2], k4[3], idx[3]);
      }
    }
  }
  __syncthreads();

  const int j0 = batch * 256 + warp * 32;
  const int nrows = min(32, J - j0);          // may be <= 0 for trailing warps
  // ---- per-lane set-up for row j0 + lane: 32 draws side by side -----------------------------
  uint32_t flags_l = 0;   // bit 0 perturb, bit 1 active, bit 2 row comes from the second parent, bits 3.. replica cap
  u32x4 mw = {0, 0, 0, 0};
  if (lane < nrows) {
    const int j = j0 + lane;
    const bool act = !a.active || a.active[j];
    int kc = a.k_cap ? a.k_cap[j] : a.k_max;
    kc = max(0, min(kc, a.k_max));
    bool mut = false, second = false;
    if (a.mode == ROWS_GENERATION) {
      if ((int)c >= a.num_elite) {
        const u32x4 x = draw(a.key, (uint32_t)j, c, a.gen, SLOT_XOVER);
        second = (x.x >> 31) != 0u;
        mw = draw(a.key, (uint32_t)j, c, a.gen, SLOT_MUTATE);
        mut = mw.x < a.thr;
      }
    } else if (a.mode == ROWS_INIT && c > 0) {
      mw = draw(a.key, (uint32_t)j, c, GEN_INIT, SLOT_INIT);
      mut = mw.x < a.thr;
    }
    flags_l = (mut ? 1u : 0u) | (act ? 2u : 0u) | (second ? 4u : 0u) | ((uint32_t)kc << 3);
  }

  // row j0 of the possible sources; per row only the offset r * NN is added
  const size_t roff0 = (size_t)j0 * NN;
  const int16_t *src_a = nullptr, *src_b = nullptr;
  if (a.mode == ROWS_GENERATION) {
    src_a = a.src + (size_t)s_parent[0] * J * NN + roff0;
    src_b = a.src + (size_t)s_parent[1] * J * NN + roff0;
  } else if (a.mode == ROWS_INIT) {
    src_a = src_b = a.src ? a.src + roff0 : nullptr;
  } else {
    src_a = src_b = a.dst + (size_t)cl * J * NN + roff0;
  }
  const int16_t *cur0 = a.cur ? a.cur + roff0 : nullptr;
  int16_t *dst0 = a.dst + (size_t)cl * J * NN + roff0;
  int16_t *row = s_row[warp];

  // Iterations are software-pipelined: the loads of the next RPI rows are issued before the
  // current ones are processed.
  // An unperturbed child row is a verbatim copy of a parent's row, whose summary (K, N, entries
  // differing from the current allocation; kept exact by the column pass) is already known:
  // such rows skip the row totals and the comparison with the current allocation.
  const bool inherit = a.mode == ROWS_GENERATION && a.summ_in != nullptr;
  const uint32_t *sin_a = inherit ? a.summ_in + (size_t)s_parent[0] * J + j0 : nullptr;
  const uint32_t *sin_b = inherit ? a.summ_in + (size_t)s_parent[1] * J + j0 : nullptr;
  uint4 raw[VPL];
  uint32_t pword = 0;
  auto fetch = [&](int r) {   // r = this lane's row within the warp's 32 (may be >= nrows)
    const uint32_t fl = __shfl_sync(0xffffffffu, flags_l, r & 31);
    const int16_t *src = (fl & 4u) ? src_b : src_a;
    const bool on = r < nrows && (fl & 2u) && src;
    const bool copy = inherit && !(fl & 1u);
    if (copy && on && sub == 0) pword = __ldg(((fl & 4u) ? sin_b : sin_a) + r);
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
      const int v = sub + LPR * q;
      raw[q] = make_uint4(0, 0, 0, 0);
      if (on && (FULL || v < row_vecs)) raw[q] = __ldg((const uint4 *)(src + (size_t)r * NN) + v);
      // the matching piece of the current allocation is read late in the iteration: pull it
      // towards L1 now, without tying up registers
      if (cur0 && !copy && r < nrows && (FULL || v < row_vecs))
        asm volatile("prefetch.global.L1 [%0];" ::"l"((const uint4 *)(cur0 + (size_t)r * NN) + v));
    }
  };
  if (nrows > 0) fetch(grp);
  // Expands the queued vectors: entry e = (vector e / 8, half e % 8), one lane per entry.  Per
  // occupant: add to the node's GPU total and distributed-job count, record it in the
  // node's occupant list.
  auto flush_queue = [&](int count) {
    __syncwarp();
    for (int e = lane; e < count * 8; e += 32) {
      const uint32_t val = ((const uint16_t *)s_qvec[warp])[e];
      if (val) {
        const uint32_t meta = s_qmeta[warp][e >> 3];
        const int n = (int)((meta >> 20) & 0x7FFu) * 8 + (e & 7);
        atomicAdd(&s_tot[n], (int)val);
        if (meta >> 31) atomicAdd(&s_el[n], 1);
        const int slot = atomicAdd(&s_cnt[n], 1);
        if (slot < OCC_SLOTS) s_occ[n * OCC_SLOTS + slot] = (meta & 0xFFFFFu) | (val << 20) | (meta & 0x80000000u);
      }
    }
    __syncwarp();
  };

  for (int r0 = 0; r0 < nrows; r0 += RPI) {
    const int r = r0 + grp;                       // this lane's row
    const bool live = r < nrows;
    const uint32_t flags = __shfl_sync(0xffffffffu, flags_l, r & 31);
    const bool act = live && (flags & 2u);
    uint4 x[VPL];
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
      const int v = sub + LPR * q;
      x[q] = make_uint4(0, 0, 0, 0);
      if (FULL || v < row_vecs) x[q] = clamp_vec(raw[q], ((const uint4 *)s_cap)[v]);
    }
    const bool copy = inherit && act && !(flags & 1u);       // uniform within the row's lanes
    const uint32_t pw = __shfl_sync(0xffffffffu, pword, grp << LPR_LOG2);
    if (r0 + RPI < nrows) fetch(r0 + RPI + grp);

    const bool compute = __any_sync(0xffffffffu, live && !copy);   // some row of this iteration needs totals
    int K = 0, N = 0;
    if (compute) {
      uint32_t part = 0;
#pragma unroll
      for (int q = 0; q < VPL; ++q) part += row_partial(x[q]);
      part = __reduce_add_sync(gmask, part);
      K = (int)(part & 0x3FFFFFu);
      N = (int)(part >> 22);
    }
    if (copy) { K = (int)(pw & 0x7FFu); N = (int)((pw >> 11) & 0x7FFu); }
    const int kc = (int)(flags >> 3);

    // rows that are perturbed or break a row cap take a detour through shared memory, one
    // row at a time with the whole warp
    unsigned need = __ballot_sync(0xffffffffu, act && !copy && sub == 0 && ((flags & 1u) || K > kc || N > a.n_max));
    while (need) {
      const int leader = __ffs(need) - 1;         // lane `leader` is sub 0 of the row's group
      need &= need - 1;
      const int g = leader >> LPR_LOG2;
      const int rr = r0 + g;
      const uint32_t rflags = __shfl_sync(0xffffffffu, flags, leader);
      int rK = __shfl_sync(0xffffffffu, K, leader), rN = __shfl_sync(0xffffffffu, N, leader);
      const int rkc = (int)(rflags >> 3);
      if (grp == g) {
#pragma unroll
        for (int q = 0; q < VPL; ++q)
          if (FULL || sub + LPR * q < row_vecs) ((uint4 *)row)[sub + LPR * q] = x[q];
      }
      __syncwarp();
      if (rflags & 1u) {
        const uint32_t m1 = __shfl_sync(0xffffffffu, mw.y, rr), m2 = __shfl_sync(0xffffffffu, mw.z, rr),
                       m3 = __shfl_sync(0xffffffffu, mw.w, rr);
        const uint32_t op = bounded(m1, 3u);
        if (op == 0u) {
          const int n = (int)bounded(m3, (uint32_t)NN);
          if (lane == 0) row[n] = (int16_t)min((int)row[n] + 1, (int)s_cap[n]);
        } else if (rN > 0) {
          const int ns = nth_occupied(row, NN, bounded(m2, (uint32_t)rN), lane);
          if (op == 1u) {
            if (lane == 0) row[ns] = (int16_t)(row[ns] - 1);
          } else {
            const int nd = (int)bounded(m3, (uint32_t)NN);
            if (nd != ns && lane == 0) {
              row[nd] = (int16_t)min((int)row[nd] + (int)row[ns], (int)s_cap[nd]);
              row[ns] = 0;
            }
          }
        }
        __syncwarp();
        rK = 0; rN = 0;
        for (int n = lane; n < NN; n += 32) { rK += row[n]; rN += row[n] > 0; }
        rK = __reduce_add_sync(0xffffffffu, rK);
        rN = __reduce_add_sync(0xffffffffu, rN);
      }
      if (rK > rkc || rN > a.n_max) {
        if (lane == 0) {
          int excess = rK - rkc;
          rK = min(rK, rkc);
          for (int n = NN - 1; n >= 0 && excess > 0; --n) {
            const int take = min((int)row[n], excess);
            row[n] = (int16_t)(row[n] - take);
            excess -= take;
          }
          int occ = 0;
          for (int n = 0; n < NN; ++n) {
            if (row[n] > 0) {
              ++occ;
              if (occ > a.n_max) { rK -= row[n]; row[n] = 0; }
            }
          }
          rN = min(occ, a.n_max);
        }
        rN = __shfl_sync(0xffffffffu, rN, 0);
        rK = __shfl_sync(0xffffffffu, rK, 0);
      }
      __syncwarp();
      if (grp == g) {
#pragma unroll
        for (int q = 0; q < VPL; ++q)
          if (FULL || sub + LPR * q < row_vecs) x[q] = ((const uint4 *)row)[sub + LPR * q];
        K = rK;
        N = rN;
      }
      __syncwarp();
    }

    // ---- store, column bookkeeping, row summary ---------------------------------------------
    const bool dist = N >= 2;
    int ndiff = 0;   // entries of this lane that differ from the current allocation
    int qn = 0;      // vectors queued by the warp in this iteration
    const int j = j0 + r;
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
      const int v = sub + LPR * q;
      const bool in = live && (FULL || v < row_vecs);
      if (in) ((uint4 *)(dst0 + (size_t)r * NN))[v] = x[q];
      // Occupied nodes are few.  Vectors with any occupant are compacted into a per-warp
      // queue (ballot + popc, no atomics) and expanded below with one lane per entry.
      if (qn > QCAP - 32) { flush_queue(qn); qn = 0; }
      const bool nz = in && (x[q].x | x[q].y | x[q].z | x[q].w) != 0u;
      const unsigned bal = __ballot_sync(0xffffffffu, nz);
      if (nz) {
        const int pos = qn + __popc(bal & ((1u << lane) - 1u));
        s_qvec[warp][pos] = x[q];
        s_qmeta[warp][pos] = (uint32_t)j | ((uint32_t)v << 20) | (dist ? 0x80000000u : 0u);   // v < 64
      }
      qn += __popc(bal);
      if (cur0 && in && !copy) {
        const uint4 cx = __ldg((const uint4 *)(cur0 + (size_t)r * NN) + v);
        const uint4 d = make_uint4(x[q].x ^ cx.x, x[q].y ^ cx.y, x[q].z ^ cx.z, x[q].w ^ cx.w);
        if ((d.x | d.y | d.z | d.w) != 0u) {
          // entries on both sides are in [0, 32767], so each half of the xor is a non-negative
          // int16 and min(half, 1) counts the halves that differ
          const uint32_t dc = __vimin_s16x2_relu(d.x, 0x00010001u) + __vimin_s16x2_relu(d.y, 0x00010001u) +
                              __vimin_s16x2_relu(d.z, 0x00010001u) + __vimin_s16x2_relu(d.w, 0x00010001u);
          ndiff += (int)((dc & 0xFFFFu) + (dc >> 16));
        }
      }
    }
    flush_queue(qn);
    qn = 0;
    if (cur0 && compute) ndiff = __reduce_add_sync(gmask, ndiff);
    if (copy) ndiff = (int)(pw >> 22);
    if (live && sub == 0) {
      const bool on = (flags & 2u) != 0u;
      a.dflag[(size_t)cl * J + j] = (on && dist) ? 1 : 0;
      // row summary for the fitness: K | N << 11 | (entries that differ from current) << 22
      const uint32_t word = on ? ((uint32_t)K | ((uint32_t)N << 11) | ((uint32_t)ndiff << 22)) : 0u;
      if (a.summ) a.summ[(size_t)cl * J + j] = word;
    }
  }

  __syncthreads();
  // ---- column partials and occupant lists of the block -------------------------------------
  const size_t base = ((size_t)cl * aa.nbatch + batch) * NN;
  for (int i = threadIdx.x; i < NN; i += blockDim.x) {
    aa.colsum[base + i] = s_tot[i];
    aa.colelig[base + i] = s_el[i];
    aa.occ_count[base + i] = s_cnt[i];
    const int cnt = min(s_cnt[i], OCC_SLOTS);
    for (int k = 0; k < cnt; ++k) aa.occ_list[(base + i) * OCC_SLOTS + k] = s_occ[i * OCC_SLOTS + k];
  }
  // The last block of the candidate to get here adds the batch partials per node and appends
  // the nodes that hold two distributed jobs or exceed their size to the work list.
  __shared__ bool s_last_block;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned prev = atomicAdd(aa.cand_ticket + cl, 1u);
    s_last_block = (prev == (unsigned)aa.nbatch - 1u);
    if (s_last_block) aa.cand_ticket[cl] = 0u;
  }
  __syncthreads();
  if (s_last_block) {
    __threadfence();
    for (int n = threadIdx.x; n < NN; n += blockDim.x) {
      int total = 0, nelig = 0;
      for (int b = 0; b < aa.nbatch; ++b) {
        total += __ldcg(aa.colsum + ((size_t)cl * aa.nbatch + b) * NN + n);
        nelig += __ldcg(aa.colelig + ((size_t)cl * aa.nbatch + b) * NN + n);
      }
      if (nelig >= 2 || total > (int)s_cap[n]) {
        const unsigned slot = atomicAdd(aa.list_count, 1u);
        aa.list[slot] = ((uint32_t)cl << 13) | (uint32_t)n;      // n < 8192, cl < 65536
      }
    }
  }
}

// Column pass: warps take nodes from the work list the row kernel built (any order: columns are
// independent) and repair them.
__global__ void __launch_bounds__(128, 4) colrepair_kernel(ColfixArgs a) {
  const int lane = threadIdx.x & 31;
  const unsigned nwarps = gridDim.x * (blockDim.x >> 5);
  const unsigned count = *a.list_count;
  const int NN = a.num_nodes;
  for (unsigned i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < count; i += nwarps) {
    const uint32_t e = a.list[i];
    const int cl = (int)(e >> 13), n = (int)(e & 0x1FFFu);
    int total = 0, nelig = 0;
    for (int b = 0; b < a.nbatch; ++b) {
      total += a.colsum[((size_t)cl * a.nbatch + b) * NN + n];
      nelig += a.colelig[((size_t)cl * a.nbatch + b) * NN + n];
    }
    const int cp = max((int)a.cap[n], 0);
    repair_column_list(a, cl, n, total, nelig, cp, lane);
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------
// A whole child per block: row pass and repair in one launch, rows of any width up to 512 nodes and any alignment
// (the dense entry points called on their own).
//
// Almost every entry of a population is zero and almost every row is copied unchanged, so a warp takes a tile
// of rows (as many as touch 160 aligned vectors of their sources and hold 1024 entries), reads each row's aligned
// vectors from the parent it comes from, and lays the tile out in shared memory, shifted to where the child lies
// between two 16-byte boundaries: zeros, and the entries of the vectors that hold something, which are queued
// (ballot + popc) and looked at one lane per entry.  Rows that are perturbed or break a row cap are
// edited there by the warp; then the tile goes out in whole vectors.  Column totals and occupant lists stay in
// shared memory, and once the block's rows are out its groups of 16 lanes decide the nodes that need repair and
// write the few entries that change.
// A child is a cluster of up to eight blocks where there are few children: every block lists the occupants that its
// rows bring, and the nodes are then decided from all their lists, over distributed shared memory.
// Bound: for large children instruction issue (55 % of the slots) and the loads' latency between two tiles, for small
// ones the chain of one block's steps.  Measured with the fitness behind it (us, before: kernels for the rows
// and for the columns): 512 children of 1024 x 256 178 -> 171, 256 of 1000 x 250 760 -> 132, 57 of 748 x 255 255 -> 45
// (83 with one block per child), 200 of 300 x 72 46 -> 29, 100 of 48 x 16 31 -> 18.5.  Tiles of 128 vectors where rows are
// not aligned: 177 us for 1000 x 250 (a tile costs the same whether it has three rows or four).
// ---------------------------------------------------------------------------------------
constexpr int CHILD_WARPS = 8;
constexpr int CHILD_TILE = 1024;        // entries a warp lays out at a time
constexpr int CHILD_OCC = 16;           // occupants a group of lanes decides; listed per node of a block: at least as many
constexpr int CHILD_CROWD = 768;        // occupants a warp decides
constexpr int CHILD_SPLIT = 8;          // blocks of a child, at most
__host__ __device__ constexpr int child_vectors(bool whole) { return whole ? 128 : 160; }   // a warp reads at a time

struct ChildArgs {
  RowsArgs r;
  ColfixArgs col;                       // for nodes with more occupants than a list holds
  const int16_t *src_lo, *src_hi;       // what may be read: [src_lo, src_hi)
  int row_vecs;                         // aligned vectors a row may touch
  int split;                            // blocks of a child: a power of two
  int occ;                              // occupants a block lists per node
  int tile_rows, chunk_rows;            // rows laid out at a time; rows whose draws are made at a time
  int *status;
};

template <bool WHOLE>
struct ChildWarp {                      // shared memory of a warp
  uint4 tile[WHOLE ? 64 : CHILD_TILE / 8 + 1];       // the tile; WHOLE: the row being edited
  uint4 qvec[child_vectors(WHOLE)];
  uint32_t qmeta[child_vectors(WHOLE)];          // row of the tile (bits 0..4) | place of its first entry in the row, + 8 unless WHOLE (8..17) | alive (31)
  uint32_t row[32];                     // of the tile: GPUs | occupied nodes << 22
  int bad[32];                          // an entry is out of range
};

static_assert(sizeof(ChildWarp<true>) >= CHILD_CROWD * 4 && sizeof(ChildWarp<false>) >= CHILD_CROWD * 4, "a crowded node's occupants");

inline size_t child_smem_bytes(int NN, int occ, bool whole) {
  return CHILD_WARPS * (whole ? sizeof(ChildWarp<true>) : sizeof(ChildWarp<false>)) + (size_t)NN * ((size_t)occ * 4 + 4 + 4 + 2);
}

// Behind the nodes' lists: GPUs placed on each; distributed jobs on it | occupants << 16.
__device__ __forceinline__ const uint32_t *child_counts(const uint32_t *s_occ, int NN, int occ) { return s_occ + (size_t)NN * occ + NN; }

// An entry of a list: job | GPUs << 16 | distributed << 31.
__device__ __forceinline__ int occupant_gpus(uint32_t e) { return (int)((e >> 16) & 0x7FFu); }
__device__ __forceinline__ int rotated(uint32_t e, uint32_t offset, int J) {
  const int r = (int)(e & 0xFFFFu) - (int)offset;
  return r < 0 ? r + J : r;
}

// The repair of a node with more occupants than a group of lanes has, by a warp: from the blocks' lists, gathered in `list`, or,
// where one of those is too short, from the column (128 children of 1024 x 8, a tenth of the rows perturbed: 24.0 us
// from lists, 32.7 from the columns where there are more than 16; three of ten, as at first, 42.9 and 51.0).
__device__ __noinline__ void repair_crowded(const ChildArgs &aa, uint32_t *list, const uint32_t *s_occ, int cl, int n, int tot, uint32_t cnt,
                                            int cap_n, uint32_t rep, int lane) {
  const int J = aa.r.J, NN = aa.r.num_nodes, count = (int)(cnt >> 16);
  const bool intf = (cnt & 0xFFFFu) >= 2u;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  bool all = count <= CHILD_CROWD;
  if (all) {
    int at = 0;
#pragma unroll 1
    for (int q = 0; q < aa.split; ++q) {
      const uint32_t *const occ = aa.split > 1 ? cluster.map_shared_rank(s_occ, q) : s_occ;
      const int here = (int)(child_counts(occ, NN, aa.occ)[n] >> 16);
      all = all && here <= aa.occ;
      for (int k = lane; k < min(here, aa.occ); k += 32)
        if (sched_index_ok(aa.status, at + k < CHILD_CROWD, SCHED_CHK_LIST)) list[at + k] = occ[n * aa.occ + k];
      at += here;
    }
    __syncwarp();
  }
  if (!all) {
    repair_column_any(aa.col, nullptr, cl, n, tot, (int)(cnt & 0xFFFFu), cap_n, lane);
    return;
  }
  const auto rot_i = [&](uint32_t e) { return rotated(e, rep & 0xFFFFu, J); };
  const auto rot_c = [&](uint32_t e) { return rotated(e, rep >> 16, J); };
  const CrowdPlaces at = crowd_places([=](int k) { return list[k]; }, count, J, tot, intf, cap_n, lane, occupant_gpus, rot_i, rot_c);
  int16_t *const column = aa.r.dst + (size_t)cl * J * NN + n;
#pragma unroll 1
  for (int k = lane; k < count; k += 32) {
    const uint32_t e = list[k];
    const int v = at.keeps(e, occupant_gpus(e), rot_i(e), rot_c(e));
    if (v != occupant_gpus(e) && sched_index_ok(aa.status, (int)(e & 0xFFFFu) < J, SCHED_CHK_NODE))
      column[(size_t)(e & 0xFFFFu) * NN] = (int16_t)v;
  }
}

// The candidate of rank c (fitness key descending, index ascending) of any number, by a block: the key from its
// top digit down by counting (four passes over the keys), then the one wanted of those that have it.  count: 288
// words of shared memory.  The work grows with the number of candidates, not with its square or the rank: a generation
// of 1024, 4096 and 16384 children of 48 x 16 with 64 elite ones 19, 55 and 199 us (842 us, 13.3 and 17.6 ms where pairs
// of keys were compared), with 4 elite ones 19, 54 and 193 (19 us, 54 us, 17.6 ms).
__device__ __noinline__ int ranked_candidate(const uint32_t *fitness_bits, int P, int c, uint32_t *count) {
  constexpr int DIGITS = 256, THREADS = CHILD_WARPS * 32;
  static_assert(THREADS == DIGITS, "a thread clears a digit's counter");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t *found = count + DIGITS, *part = found + 4;       // digit, rank among its keys; equal keys by warp; the candidate
  uint32_t key = 0u, known = 0u, rank = (uint32_t)c;
#pragma unroll 1
  for (int shift = 24; shift >= 0; shift -= 8) {
    count[tid] = 0u;
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < P; i += THREADS) {
      const uint32_t k = order_key(__ldg(fitness_bits + i));
      if ((k & known) == key) atomicAdd(&count[(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (warp == 0) {                    // eight digits a lane, the largest first
      uint32_t sum = 0u, upto;
#pragma unroll
      for (int d = 0; d < 8; ++d) sum += count[255 - 8 * lane - d];
      upto = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, upto, off);
        if (lane >= off) upto += u;
      }
      if (rank >= upto - sum && rank < upto) {
        uint32_t left = rank - (upto - sum), digit = 255u - 8u * (uint32_t)lane;
#pragma unroll 1
        while (left >= count[digit]) left -= count[digit--];
        found[0] = digit;
        found[1] = left;
      }
    }
    __syncthreads();
    key |= found[0] << shift;
    known |= 255u << shift;
    rank = found[1];
  }
  // of the candidates with this key the rank-th: a warp counts those of consecutive ones
  const int per = ((P + THREADS - 1) / THREADS) * 32, lo = min(P, warp * per), hi = min(P, lo + per);
  uint32_t mine = 0u;
#pragma unroll 4
  for (int i = lo; i < hi; i += 32)
    mine += (uint32_t)__popc(__ballot_sync(0xffffffffu, i + lane < hi && order_key(__ldg(fitness_bits + min(i + lane, P - 1))) == key));
  if (lane == 0) part[warp] = mine;
  __syncthreads();
  uint32_t before = 0u;
#pragma unroll 1
  for (int w = 0; w < warp; ++w) before += part[w];
  if (rank >= before && rank < before + mine) {
    uint32_t left = rank - before;
#pragma unroll 1
    for (int i = lo; i < hi; i += 32) {
      const unsigned m = __ballot_sync(0xffffffffu, i + lane < hi && order_key(__ldg(fitness_bits + min(i + lane, P - 1))) == key);
      const uint32_t here = (uint32_t)__popc(m);
      if (left < here) {
        if (((m >> lane) & 1u) && (uint32_t)__popc(m & ((1u << lane) - 1u)) == left) found[2] = (uint32_t)(i + lane);
        break;
      }
      left -= here;
    }
  }
  __syncthreads();
  return (int)found[2];
}

// WHOLE: rows are whole vectors on 16-byte boundaries.  Their vectors go straight out again, and only a row
// that is edited (perturbed, over a cap, an entry out of range) is laid out, from its queued vectors, and written once more.
template <bool WHOLE>
__global__ void __launch_bounds__(CHILD_WARPS * 32, WHOLE ? 4 : 3) child_kernel(const __grid_constant__ ChildArgs aa) {
  extern __shared__ __align__(16) unsigned char child_smem[];
  const RowsArgs &a = aa.r;
  const int NN = a.num_nodes, J = a.J, P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ChildWarp<WHOLE> &w = ((ChildWarp<WHOLE> *)child_smem)[warp];
  uint32_t *s_occ = (uint32_t *)(child_smem + CHILD_WARPS * sizeof(ChildWarp<WHOLE>));   // job | GPUs << 16 | distributed << 31
  int32_t *s_tot = (int32_t *)(s_occ + (size_t)NN * aa.occ);                         // GPUs placed on the node
  uint32_t *s_cnt = (uint32_t *)(s_tot + NN);                                        // distributed jobs on it | occupants << 16
  int16_t *s_cap = (int16_t *)(s_cnt + NN);
  __shared__ int s_parent[2];
  // a cluster of `split` blocks to a child; gw: this warp among all of them
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int split = aa.split, part = (int)blockIdx.x & (split - 1), cl = (int)blockIdx.x / split;
  const int gw = part * CHILD_WARPS + warp, nwarps = split * CHILD_WARPS;
  const uint32_t c = a.first_cand + (uint32_t)cl, round = round_of(a.key);
  const bool bred = a.mode == ROWS_GENERATION && (int)c >= a.num_elite;
  for (int i = tid; i < NN; i += blockDim.x) {
    s_tot[i] = 0;
    s_cnt[i] = 0u;
    s_cap[i] = (int16_t)max((int)a.cap[i], 0);
  }

  // ---- the draws of this warp's next rows, a lane each -----------------------------------------------
  bool act_l = false, mut_l = false, sec_l = false;
  int kc_l = 0;
  u32x4 mw = {0, 0, 0, 0};
  auto draw_rows = [&](int j0) {
    act_l = mut_l = sec_l = false;
    const int j = j0 + lane;
    if (lane >= aa.chunk_rows || j >= J) return;
    act_l = !a.active || a.active[j];
    kc_l = max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max));
    if (bred) {
      uint32_t x;
      draw_two(a.key.k0, round, (uint32_t)j, c, a.gen, SLOT_XOVER, SLOT_MUTATE, x, mw);
      sec_l = (x >> 31) != 0u;
      mut_l = mw.x < a.thr;
    } else if (a.mode == ROWS_INIT && c > 0u) {
      mw = draw_one(a.key.k0, round, (uint32_t)j, c, GEN_INIT, SLOT_INIT);
      mut_l = mw.x < a.thr;
    }
  };
  draw_rows(gw * aa.chunk_rows);

  // ---- parents (generation mode): the candidate of its rank for an elite child, else the better-ranked of two
  // random pairs ---------------------------------------------------------------------------------------
  if (bred) {
    if (warp == 0) {
      const u32x4 sel = draw_one(a.key.k0, round, 0u, c, a.gen, SLOT_SELECT);
      const int i = (int)bounded(lane == 0 ? sel.x : lane == 1 ? sel.y : lane == 2 ? sel.z : sel.w, (uint32_t)P);
      const uint32_t k = order_key(__ldg(a.fitness_bits + i));
      const int io = __shfl_down_sync(0xffffffffu, i, 1);
      const uint32_t ko = __shfl_down_sync(0xffffffffu, k, 1);
      if (lane == 0 || lane == 2) s_parent[lane >> 1] = tournament_winner(k, i, ko, io);
    }
  } else if (a.mode == ROWS_GENERATION) {
    const int i = ranked_candidate(a.fitness_bits, P, (int)c, (uint32_t *)child_smem);
    if (tid == 0) s_parent[0] = s_parent[1] = i;
  }
  __syncthreads();

  const size_t mat = (size_t)J * NN;
  int16_t *child = a.dst + (size_t)cl * mat;
  const int16_t *src_a = a.src, *src_b;           // NULL: the rows start empty
  if (a.mode == ROWS_GENERATION) {
    const bool found = sched_index_ok(aa.status, (unsigned)s_parent[0] < (unsigned)P && (unsigned)s_parent[1] < (unsigned)P, SCHED_CHK_SLOT);
    src_b = a.src + (found ? (size_t)s_parent[1] * mat : 0);
    src_a += found ? (size_t)s_parent[0] * mat : 0;
  } else {
    if (a.mode == ROWS_REPAIR) src_a = child;
    src_b = src_a;
  }
  auto add_occupant = [&](int j, int n, int v, bool dist) {
    if (!sched_index_ok(aa.status, n < NN && j < J && v <= 2047, SCHED_CHK_NODE)) return;
    atomicAdd(&s_tot[n], v);
    const uint32_t k = atomicAdd(&s_cnt[n], (dist ? 1u : 0u) | (1u << 16)) >> 16;
    if (k < (uint32_t)aa.occ) s_occ[n * aa.occ + k] = (uint32_t)j | ((uint32_t)v << 16) | (dist ? 0x80000000u : 0u);
  };
  constexpr int B = child_vectors(WHOLE) / 32;
  int16_t *tile = (int16_t *)w.tile;
  // the lane's vectors of a tile: row | place in the row << 8 (that of its first entry, before the row's skew)
  uint32_t at_q[B];
  {
    const uint32_t inv = (65536u + (uint32_t)aa.row_vecs - 1u) / (uint32_t)aa.row_vecs;   // t / row_vecs = t * inv >> 16 (t < 160)
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const uint32_t t = (uint32_t)(q * 32 + lane), r = (t * inv) >> 16;
      at_q[q] = min(r, 31u) | ((8u * (t - r * (uint32_t)aa.row_vecs)) << 8) | (r < (uint32_t)aa.tile_rows ? 0u : 0x80000000u);
    }
  }

#pragma unroll 1
  for (int j0 = gw * aa.chunk_rows; j0 < J; j0 += nwarps * aa.chunk_rows) {
    const int nrows = min(aa.chunk_rows, J - j0);
    const unsigned act_mask = __ballot_sync(0xffffffffu, act_l), sec_mask = __ballot_sync(0xffffffffu, sec_l);
    const unsigned mut_mask = __ballot_sync(0xffffffffu, mut_l && act_l);
#pragma unroll 1
    for (int r0 = 0; r0 < nrows; r0 += aa.tile_rows) {
      const int rows = min(aa.tile_rows, nrows - r0), ent = rows * NN, jt = j0 + r0;
      int16_t *out = child + (size_t)jt * NN;
      const int skew = WHOLE ? 0 : (int)(((uintptr_t)out & 15) >> 1);      // entry e of the tile lies at skew + e
      const int out_vecs = (skew + ent + 7) >> 3;
      // ---- in: four or five vectors a lane, queued if they hold anything ---------------------------------
      const int16_t *const from_a = src_a + (size_t)jt * NN, *const from_b = src_b + (size_t)jt * NN;
      const unsigned load_rows = src_a ? act_mask >> r0 : 0u, sec_rows = sec_mask >> r0;
      uint4 x[B];
      uint32_t meta[B];
      if (WHOLE) {
#pragma unroll
        for (int q = 0; q < B; ++q) {
          const uint32_t r = at_q[q] & 31u;
          x[q] = make_uint4(0u, 0u, 0u, 0u);
          meta[q] = at_q[q] | 0x80000000u;
          if (q * 32 + lane < out_vecs && ((load_rows >> r) & 1u))
            x[q] = *((const uint4 *)(((sec_rows >> r) & 1u) ? from_b : from_a) + (q * 32 + lane));
        }
      } else {
        // (vectors reach up to seven entries beyond their rows: not beyond the sources)
        const bool inside = from_a - 7 >= aa.src_lo && from_b - 7 >= aa.src_lo && from_a + ent + 7 <= aa.src_hi &&
                            from_b + ent + 7 <= aa.src_hi;
        const int skew_a = (int)((uintptr_t)from_a >> 1), skew_b = (int)((uintptr_t)from_b >> 1);
#pragma unroll
        for (int q = 0; q < B; ++q) {
          const int r = (int)(at_q[q] & 31u), first = r * NN;
          const bool sec = (sec_rows >> r) & 1u;
          const int e = (int)((at_q[q] >> 8) & 0x3FFu) - (((sec ? skew_b : skew_a) + first) & 7);
          x[q] = make_uint4(0u, 0u, 0u, 0u);
          meta[q] = (uint32_t)r | ((uint32_t)(e + 8) << 8) | 0x80000000u;
          if ((int)at_q[q] >= 0 && r < rows && e < NN && ((load_rows >> r) & 1u)) {
            const int16_t *const p = (sec ? from_b : from_a) + first + e;
            if (inside || (p >= aa.src_lo && p + 8 <= aa.src_hi)) {
              x[q] = *(const uint4 *)p;
            } else {
              uint32_t y[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
              for (int h = max(0, -e); h < 8 && e + h < NN; ++h)
                y[h >> 1] |= (uint32_t)(uint16_t)p[h] << (16 * (h & 1));
              x[q] = make_uint4(y[0], y[1], y[2], y[3]);
            }
          }
        }
      }
      if (!WHOLE)
        for (int v = lane; v < out_vecs; v += 32) w.tile[v] = make_uint4(0u, 0u, 0u, 0u);
      w.row[lane] = 0u;
      if (WHOLE) w.bad[lane] = 0;
      int qn = 0;
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const bool nz = (x[q].x | x[q].y | x[q].z | x[q].w) != 0u;
        const unsigned bal = __ballot_sync(0xffffffffu, nz);
        if (nz) {
          const int pos = qn + __popc(bal & ((1u << lane) - 1u));
          w.qvec[pos] = x[q];
          w.qmeta[pos] = meta[q];
        }
        qn += __popc(bal);
        if (WHOLE && q * 32 + lane < out_vecs) ((uint4 *)out)[q * 32 + lane] = x[q];
      }
      __syncwarp();
      // ---- first look: entries (those of the vector's own row, forced into [0, node size]) to their places, the
      // rows' K and N ------------------------------------------------------------------------------------
      for (int e = lane; e < qn * 8; e += 32) {
        const int val = (int)((const int16_t *)w.qvec)[e];
        const uint32_t m = w.qmeta[e >> 3];
        const int r = (int)(m & 31u), n = (int)((m >> 8) & 0x3FFu) - (WHOLE ? 0 : 8) + (e & 7);
        if (WHOLE ? val != 0 : val > 0 && n >= 0 && n < NN) {
          const int cv = min(max(val, 0), (int)s_cap[n]);
          if (!WHOLE) tile[skew + r * NN + n] = (int16_t)cv;
          else if (cv != val) w.bad[r] = 1;
          if (cv > 0) atomicAdd(&w.row[r], (uint32_t)cv | (1u << 22));
        }
      }
      __syncwarp();
      // ---- rows that are perturbed or break a row cap: edited where they lie ----------------------------
      bool need_l = false;
      const int kc_r = __shfl_sync(0xffffffffu, kc_l, (r0 + lane) & 31);      // the cap of the tile's lane-th row
      if (lane < rows)
        need_l = ((act_mask >> (r0 + lane)) & 1u) &&
                 (((mut_mask >> (r0 + lane)) & 1u) || (int)(w.row[lane] & 0x3FFFFFu) > kc_r || (int)(w.row[lane] >> 22) > a.n_max ||
                  (WHOLE && w.bad[lane]));
      unsigned need = __ballot_sync(0xffffffffu, need_l);
#pragma unroll 1
      while (need) {
        const int rl = __ffs(need) - 1, rr = r0 + rl;
        need &= need - 1;
        int16_t *row = WHOLE ? tile : tile + skew + rl * NN;
        if (WHOLE) {                    // laid out from its vectors
          for (int v = lane; v < aa.row_vecs; v += 32) w.tile[v] = make_uint4(0u, 0u, 0u, 0u);
          __syncwarp();
          for (int e = lane; e < qn * 8; e += 32) {
            const int n = (int)((w.qmeta[e >> 3] >> 8) & 0x3FFu) + (e & 7);
            if ((w.qmeta[e >> 3] & 31u) == (uint32_t)rl)
              row[n] = (int16_t)min(max((int)((const int16_t *)w.qvec)[e], 0), (int)s_cap[n]);
          }
          __syncwarp();
        }
        int rK = (int)(w.row[rl] & 0x3FFFFFu), rN = (int)(w.row[rl] >> 22);
        if ((mut_mask >> rr) & 1u) {
          const uint32_t m1 = __shfl_sync(0xffffffffu, mw.y, rr), m2 = __shfl_sync(0xffffffffu, mw.z, rr),
                         m3 = __shfl_sync(0xffffffffu, mw.w, rr);
          const uint32_t op = bounded(m1, 3u);
          if (op == 0u) {
            const int n = (int)bounded(m3, (uint32_t)NN);
            if (lane == 0) row[n] = (int16_t)min((int)row[n] + 1, (int)s_cap[n]);
          } else if (rN > 0) {
            int ns = nth_occupied(row, NN, bounded(m2, (uint32_t)rN), lane);
            if (!sched_index_ok(aa.status, ns >= 0 && ns < NN, SCHED_CHK_NODE)) ns = 0;
            if (op == 1u) {
              if (lane == 0) row[ns] = (int16_t)(row[ns] - 1);
            } else {
              const int nd = (int)bounded(m3, (uint32_t)NN);
              if (nd != ns && lane == 0) {
                row[nd] = (int16_t)min((int)row[nd] + (int)row[ns], (int)s_cap[nd]);
                row[ns] = 0;
              }
            }
          }
          __syncwarp();
          rK = 0; rN = 0;
          for (int n = lane; n < NN; n += 32) { rK += row[n]; rN += row[n] > 0; }
          rK = __reduce_add_sync(0xffffffffu, rK);
          rN = __reduce_add_sync(0xffffffffu, rN);
        }
        const int rkc = __shfl_sync(0xffffffffu, kc_l, rr);
        if (rK > rkc || rN > a.n_max) {
          if (lane == 0) {
            int excess = rK - rkc;
            for (int n = NN - 1; n >= 0 && excess > 0; --n) {
              const int take = min((int)row[n], excess);
              row[n] = (int16_t)(row[n] - take);
              excess -= take;
            }
            int occ = 0;
            for (int n = 0; n < NN; ++n)
              if (row[n] > 0 && ++occ > a.n_max) row[n] = 0;
            rN = min(occ, a.n_max);
          }
          rN = __shfl_sync(0xffffffffu, rN, 0);
          __syncwarp();
        }
        // its queued vectors are dropped, its occupants added from where it lies
        if (lane == 0) w.row[rl] = (uint32_t)rN << 22;
        for (int e = lane; e < qn; e += 32)
          if ((w.qmeta[e] & 31u) == (uint32_t)rl) w.qmeta[e] &= 0x7FFFFFFFu;
        for (int n = lane; n < NN; n += 32)
          if (row[n] > 0) add_occupant(jt + rl, n, (int)row[n], rN >= 2);
        if (WHOLE)
          for (int v = lane; v < aa.row_vecs; v += 32) ((uint4 *)(out + (size_t)rl * NN))[v] = w.tile[v];
        __syncwarp();
      }
      // ---- second look: column totals and occupant lists; out -------------------------------------------
      for (int e = lane; e < qn * 8; e += 32) {
        const int val = (int)((const int16_t *)w.qvec)[e];
        const uint32_t m = w.qmeta[e >> 3];
        const int r = (int)(m & 31u), n = (int)((m >> 8) & 0x3FFu) - (WHOLE ? 0 : 8) + (e & 7);
        if ((m >> 31) && val > 0 && (WHOLE || (n >= 0 && n < NN))) {
          const int cv = min(val, (int)s_cap[n]);
          if (cv > 0) add_occupant(jt + r, n, cv, (w.row[r] >> 23) != 0u);
        }
      }
      if (!WHOLE) {
        for (int v = lane + (skew ? 1 : 0); 8 * v + 8 <= skew + ent; v += 32) ((uint4 *)(out - skew))[v] = w.tile[v];
        // the two vectors shared with the rows next to the tile, an entry each
        const int i = lane < 8 ? lane : ((skew + ent) & ~7) + (lane & 7);
        if (lane < 16 && i >= skew && i < skew + ent && (lane < 8 ? skew != 0 : (skew == 0 || i >= 8))) out[i - skew] = tile[i];
      }
      if (lane < rows) a.dflag[(size_t)cl * J + jt + lane] = (w.row[lane] >> 23) != 0u ? 1 : 0;
      __syncwarp();
    }
    draw_rows(j0 + nwarps * aa.chunk_rows);
  }
  if (split > 1) cluster.sync();
  else __syncthreads();

  // ---- repair: the nodes are dealt out to all warps; a lane looks at a node, groups of 16 lanes decide those
  // that hold two distributed jobs or more GPUs than they have, from the occupants that the child's blocks have
  // listed; those with more than a group has lanes by a warp each --------------------------------------
  auto of_part = [&](auto *p, int q) { return split > 1 ? cluster.map_shared_rank(p, q) : p; };
#pragma unroll 1
  for (int n0 = gw; n0 < NN; n0 += 32 * nwarps) {
    const int n_l = n0 + lane * nwarps;
    int tot_l = 0, cap_l = 0;
    uint32_t cnt_l = 0u;                // (a sum over all blocks: at most J of each, below 65536)
    if (n_l < NN) {
      cap_l = (int)s_cap[n_l];
#pragma unroll 1
      for (int q = 0; q < split; ++q) {
        tot_l += of_part(s_tot, q)[n_l];
        cnt_l += of_part(s_cnt, q)[n_l];
      }
    }
    const bool bad = (cnt_l & 0xFFFFu) >= 2u || tot_l > cap_l;
    unsigned todo = __ballot_sync(0xffffffffu, bad);
    if (todo == 0u) continue;
    uint32_t rep_l = 0u;                // the two rotation offsets
    if (bad) {
      uint32_t x;
      u32x4 y;
      draw_two(a.key.k0, round, (uint32_t)n_l, c, a.gen, SLOT_REPAIR_INTF, SLOT_REPAIR_CAP, x, y);
      rep_l = bounded(x, (uint32_t)J) | (bounded(y.x, (uint32_t)J) << 16);
    }
    __syncwarp();
#pragma unroll 1
    while (todo) {
      const int b0 = __ffs(todo) - 1;
      todo &= todo - 1;
      int b1 = -1;
      if (todo) { b1 = __ffs(todo) - 1; todo &= todo - 1; }
      const int b = (lane & 16) ? b1 : b0, sub = lane & 15, from = max(b, 0);
      const uint32_t rep = __shfl_sync(0xffffffffu, rep_l, from), cnt = __shfl_sync(0xffffffffu, cnt_l, from);
      const int tot = __shfl_sync(0xffffffffu, tot_l, from), cap_n = __shfl_sync(0xffffffffu, cap_l, from);
      const int n = n0 + from * nwarps, count = b >= 0 ? (int)(cnt >> 16) : 0;
      const bool listed = count <= CHILD_OCC, have = listed && sub < count;
      uint32_t e = 0u;
      if (have) {                       // the sub-th of the blocks' lists, one behind the other
        int q = 0, k = sub;
#pragma unroll 1
        for (; q < split - 1; ++q) {
          const int here = (int)(of_part(s_cnt, q)[n] >> 16);
          if (k < here) break;
          k -= here;
        }
        e = of_part(s_occ, q)[n * aa.occ + k];
      }
      const int j = (int)(e & 0xFFFFu), v_old = (int)((e >> 16) & 0x7FFu);
      int ri = j - (int)(rep & 0xFFFFu), rc = have ? j - (int)(rep >> 16) : 0x3fffffff;
      if (ri < 0) ri += J;
      if (rc < 0) rc += J;
      const int most = max(__shfl_sync(0xffffffffu, count, 0), __shfl_sync(0xffffffffu, count, 16));
      const int v = decide(v_old, (e >> 31) != 0u, have, min(most, CHILD_OCC), (cnt & 0xFFFFu) >= 2u, tot, cap_n, ri, rc);
      if (have && v != v_old && sched_index_ok(aa.status, j < J && n < NN, SCHED_CHK_NODE)) child[(size_t)j * NN + n] = (int16_t)v;
#pragma unroll 1
      for (unsigned walk = __ballot_sync(0xffffffffu, !listed && sub == 0); walk; walk &= walk - 1) {
        const int l = __ffs(walk) - 1;
        repair_crowded(aa, (uint32_t *)&w, s_occ, cl, __shfl_sync(0xffffffffu, n, l), __shfl_sync(0xffffffffu, tot, l),
                       __shfl_sync(0xffffffffu, cnt, l), __shfl_sync(0xffffffffu, cap_n, l), __shfl_sync(0xffffffffu, rep, l), lane);
        __syncwarp();
      }
    }
  }
  if (split > 1) cluster.sync();        // (the other blocks may still read this one's lists)
}

int launch_rows(sched_ctx *ctx, RowsArgs &a) {
  const long long warps = (long long)a.count * a.J;
  if (warps == 0) return SCHED_OK;
  const int wpb = 8;
  const size_t smem = (size_t)wpb * ((a.num_nodes + 7) & ~7) * sizeof(int16_t);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) {
      set_error(ctx, "cudaFuncSetAttribute failed: %s", cudaGetErrorString(e));
      return SCHED_ERR_CUDA;
    }
  }
  const long long blocks = (warps + wpb - 1) / wpb;
  {
  TimedLaunch tl_(ctx, KK_ROWS);
  rows_kernel<<<(unsigned)blocks, wpb * 32, smem, ctx->stream>>>(a);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

int launch_cols(sched_ctx *ctx, const RngKey &key, int16_t *pop, int count, uint32_t first_cand, uint32_t gen) {
  if (count == 0 || ctx->cfg.num_jobs == 0) return SCHED_OK;
  ColsArgs a;
  a.pop = pop; a.dflag = ctx->d_dflag; a.cap = ctx->d_cap;
  a.J = ctx->cfg.num_jobs; a.num_nodes = ctx->cfg.num_nodes;
  a.gen = gen; a.key = key;
  for (int first = 0; first < count; first += 65535) {
    const int n = min(65535, count - first);
    a.count = n;
    a.first_cand = first_cand + (uint32_t)first;
    a.pop = pop + (size_t)first * a.J * a.num_nodes;
    a.dflag = ctx->d_dflag + (size_t)first * a.J;
    dim3 grid((unsigned)((a.num_nodes + 127) / 128), (unsigned)n);
    { TimedLaunch tl_(ctx, KK_COLS); cols_kernel<<<grid, 128, 0, ctx->stream>>>(a); }
    SCHED_LAUNCH_CHECK(ctx);
  }
  return SCHED_OK;
}

bool whole_rows(const RowsArgs &a) { return a.num_nodes % 8 == 0 && (((uintptr_t)a.dst | (uintptr_t)a.src) & 15) == 0; }

int child_occupants(const sched_ctx *ctx, const RowsArgs &a) {
  return std::min(CHILD_CROWD, listed_occupants(ctx, a.mode == ROWS_REPAIR ? ctx->cfg.thr_mutate : a.thr, 256 * CHILD_OCC / a.num_nodes));
}

// Places for blocks on the GPU: three an SM (registers), four where rows are whole and their lists leave the memory for it.  Four
// pay where a block has much to copy (128 children of 1024 x 256 with three 54 us, with four 44); small ones they only
// cut up further (repair of 64 children of 1024 x 8 8.7 us, 10.7).
long long child_places(const sched_ctx *ctx, const RowsArgs &a) {
  const bool whole = whole_rows(a);
  const size_t smem = child_smem_bytes(a.num_nodes, child_occupants(ctx, a), whole) + 1024;
  const long long most = whole && (long long)a.J * a.num_nodes >= 1 << 17 ? 4 : 3;
  return std::min<long long>(most, 228 * 1024 / smem) * ctx->num_sms;
}

// Blocks of a child: more than one while that leaves none of them without a place and every warp a few rows.
int child_split(const sched_ctx *ctx, const RowsArgs &a, int count) {
  const long long places = child_places(ctx, a);
  int split = 1;
  while (split < CHILD_SPLIT && (long long)count * split * 2 <= places && split * 2 * CHILD_WARPS * 4 <= a.J) split *= 2;
  return split;
}

// Row pass and repair in one launch (child_kernel).
int launch_children(sched_ctx *ctx, const RowsArgs &a, int count, uint32_t first_cand, uint32_t gen) {
  const int NN = a.num_nodes;
  ChildArgs ca = {};
  ca.r = a;
  ca.status = ctx->d_status;
  ca.col.pop = a.dst; ca.col.dflag = a.dflag; ca.col.cap = a.cap;
  ca.col.J = a.J; ca.col.num_nodes = NN;
  ca.col.gen = gen; ca.col.first_cand = first_cand; ca.col.key = a.key;
  const size_t mat = (size_t)a.J * NN;
  ca.src_lo = a.src;
  ca.src_hi = a.src + mat * (a.mode == ROWS_GENERATION ? a.P : a.mode == ROWS_REPAIR ? count : a.src ? 1 : 0);
  const bool whole = whole_rows(a);
  ca.split = child_split(ctx, a, count);
  ca.occ = child_occupants(ctx, a);
  ca.row_vecs = whole ? NN / 8 : (NN + 14) / 8;
  const int warps = CHILD_WARPS * ca.split, turns = (a.J + 32 * warps - 1) / (32 * warps);
  ca.chunk_rows = (a.J + warps * turns - 1) / (warps * turns);
  ca.tile_rows = std::min(ca.chunk_rows, whole ? child_vectors(true) / ca.row_vecs
                                               : std::min(child_vectors(false) / ca.row_vecs, CHILD_TILE / NN));
  void (*const kernel)(ChildArgs) = whole ? child_kernel<true> : child_kernel<false>;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)count * (unsigned)ca.split);
  lc.blockDim = dim3(CHILD_WARPS * 32);
  lc.dynamicSmemBytes = child_smem_bytes(NN, ca.occ, whole);
  lc.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ca.split;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1u;
  lc.attrs = attr;
  lc.numAttrs = ca.split > 1 ? 1 : 0;
  if (lc.dynamicSmemBytes > 47 * 1024)        // (48 KB need no asking for, the static ones among them)
    SCHED_CUDA_CHECK(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lc.dynamicSmemBytes));
  {
    TimedLaunch tl_(ctx, KK_ROWS);
    SCHED_CUDA_CHECK(ctx, cudaLaunchKernelEx(&lc, kernel, ca));
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

// Whether rows of whole vectors are quicker on the batched kernels (a block per 256 rows of a child) than in
// child_kernel, whose blocks are at most eight per child.  us, child_kernel against the batched kernels:
//  * so few children that SMs stay empty, with many entries for each block (what a row costs beside its nodes is
//    worth some 64 of them in a repair, 192 where rows are perturbed): generation of 1 child of 2048 x 256 25 / 32, 4096 39 / 32,
//    32768 177 / 57; 16 children of 2048 x 512 41 / 48, 4096 x 512 75 / 56, 4096 x 128 33 / 33, 8192 x 128 44 / 39; repair of
//    1 of 4096 x 256 26 / 23, 4 of 8192 x 64 17 / 17, 16384 x 64 27 / 20, 16 of 2048 x 512 31 / 37, 4096 x 512 50 / 42;
//  * rows of more than 256 nodes, when a power of two of blocks a child leaves a third of the places empty: generation of 128
//    children of 1024 x 512 89 / 76, 4096 x 512 259 / 245; 200 of 1024 x 512, which fill them, 102 / 117.
// Not where nodes are crowded: the batched kernels list eight occupants a node and 256 rows, and 32 in all (generation of 16
// children of 32768 x 8 74 / 279, x 64 103 / 93).
bool batched_rows_pay(const sched_ctx *ctx, const RowsArgs &a, int count) {
  const int split = child_split(ctx, a, count), rows = (a.J + split - 1) / split, NN = a.num_nodes;
  const bool still = a.mode == ROWS_REPAIR || (a.mode == ROWS_INIT && count == 1);       // no row is perturbed
  const uint32_t thr = a.mode == ROWS_REPAIR ? ctx->cfg.thr_mutate : still ? 0u : a.thr;
  const double crowd = a.J * (thr / 4294967296.0) * (2.0 / 3.0) / NN;      // (two of three perturbed rows take a node)
  if (crowd + 2.0 * std::sqrt(crowd) > 30.0) return false;
  if (2LL * count * split < 3LL * ctx->num_sms) return (long long)rows * (NN + (still ? 64 : 192)) >= (still ? 155000 : 190000);
  return NN > 256 && (long long)count * split * 10 < child_places(ctx, a) * 7 && (long long)count * a.J * NN >= 60000000;
}

size_t batched_scratch(const RowsArgs &a, int count) { return (size_t)count * ((a.J + 255) / 256) * a.num_nodes; }

// What the batched kernels need beside the matrices. child_kernel does without: a call that could take either is not refused
// for the lack of it, nor while its stream is captured.
bool have_batched_scratch(sched_ctx *ctx, const RowsArgs &a, int count) {
  if (batched_scratch(a, count) <= ctx->col_cap) return true;
  cudaStreamCaptureStatus capture;
  if (cudaStreamIsCapturing(ctx->stream, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone &&
      ensure_colscratch(ctx, batched_scratch(a, count)) == SCHED_OK)
    return true;
  cudaGetLastError();
  return false;
}

// Whether children of a few rows are quicker on the general kernels, a warp a row and a thread a node, than with a block each:
// where there are many more of them than places, and no ranks to find.  us, child_kernel against the pair: initial population of
// 8000 children of 4 x 3 74 / 25, 16 x 3 97 / 64, 24 x 20 117 / 96, 24 x 41 123 / 107, 16 x 301 132 / 109, 2000 of 8 x 20 28 / 17;
// 600 of 20 x 75 17 / 19, 8000 of 20 x 301 faster in child_kernel, too.
bool tiny_children(const sched_ctx *ctx, const RowsArgs &a, int count) {
  return a.mode != ROWS_GENERATION && !whole_rows(a) && count > 7 * ctx->num_sms && a.J <= 24 && a.J * (a.num_nodes + 300) <= 9700;
}

// Row pass + column pass of `count` candidates.  Rounds on dense matrices want per-row summaries: rows of whole
// 16-byte vectors take the batched kernels with fused column sums.  Without summaries every width takes a block (or
// a few) per child where no other kernels pay, up to 512 nodes (a tile holds two rows), sizes <= 2047 (an occupant's word) and
// 65535 jobs (a node's counters); with more jobs, rows of whole vectors take the batched kernels, too (up to 2^20 jobs: an occupant's
// word there).  What is left takes the general warp-per-row / thread-per-column pair.
int launch_rows_cols(sched_ctx *ctx, RowsArgs &a, int16_t *pop, int count, uint32_t first_cand, uint32_t gen) {
  if (count == 0 || a.J == 0) return SCHED_OK;
  const int NN = a.num_nodes;
  const bool aligned = ((((uintptr_t)a.dst | (uintptr_t)a.src | (uintptr_t)a.cur) & 15) == 0);
  const bool fused = (NN % 8 == 0) && NN <= 512 && aligned && ctx->cap_max <= 2047 && count <= 65535 &&
                     a.J <= (1 << 20);
  ctx->summ_valid = fused && a.summ != nullptr;
  if (!ctx->summ_valid && NN <= 512 && ctx->cap_max <= 2047 && a.J <= 65535 && !tiny_children(ctx, a, count) &&
      !(fused && batched_rows_pay(ctx, a, count) && have_batched_scratch(ctx, a, count)))
    return launch_children(ctx, a, count, first_cand, gen);
  if (!fused) {
    if (a.mode == ROWS_GENERATION) {
      {
        TimedLaunch tl_(ctx, KK_RANK);
        rank_kernel<<<(a.P + 127) / 128, 128, 0, ctx->stream>>>(a.fitness_bits, a.P, ctx->d_rank, ctx->d_order);
      }
      SCHED_LAUNCH_CHECK(ctx);
    }
    int rc = launch_rows(ctx, a);
    if (rc != SCHED_OK) return rc;
    return launch_cols(ctx, a.key, pop, count, first_cand, gen);
  }
  const int nbatch = (a.J + 255) / 256;
  int rc = ensure_colscratch(ctx, batched_scratch(a, count));
  if (rc != SCHED_OK) return rc;
  Rows2Args aa;
  aa.r = a;
  aa.colsum = ctx->d_colsum; aa.colelig = ctx->d_colelig; aa.nbatch = nbatch;
  aa.list_count = ctx->d_colcount; aa.list = ctx->d_collist; aa.cand_ticket = ctx->d_rowticket;
  aa.occ_count = ctx->d_occcount; aa.occ_list = ctx->d_occlist;
  dim3 grid((unsigned)nbatch, (unsigned)count);
  SCHED_CUDA_CHECK(ctx, cudaMemsetAsync(ctx->d_colcount, 0, sizeof(unsigned int), ctx->stream));
  {
    TimedLaunch tl_(ctx, KK_ROWS);
    // about four vectors per lane: several loads in flight and the per-row overhead shared
    const int row_vecs = NN / 8;
    int lpr_log2 = 0;
    while ((4 << lpr_log2) < row_vecs && lpr_log2 < 5) ++lpr_log2;
    aa.lpr_log2 = lpr_log2;
    const int vpl = (row_vecs + (1 << lpr_log2) - 1) >> lpr_log2;
    const bool full = (vpl << lpr_log2) == row_vecs && (vpl == 1 || vpl == 2 || vpl == 4);
#define ROWS2(L, V)                                                      \
  do {                                                                   \
    if (full) rows2_kernel<L, V, true><<<grid, 256, 0, ctx->stream>>>(aa); \
    else rows2_kernel<L, V, false><<<grid, 256, 0, ctx->stream>>>(aa);     \
  } while (0)
    if (lpr_log2 == 0) {
      if (vpl <= 1) ROWS2(0, 1);
      else if (vpl == 2) ROWS2(0, 2);
      else ROWS2(0, 4);
    } else if (lpr_log2 == 1) ROWS2(1, 4);
    else if (lpr_log2 == 2) ROWS2(2, 4);
    else if (lpr_log2 == 3) ROWS2(3, 4);
    else ROWS2(4, 4);
#undef ROWS2
  }
  SCHED_LAUNCH_CHECK(ctx);
  ColfixArgs f;
  f.pop = pop; f.dflag = ctx->d_dflag; f.cap = ctx->d_cap;
  f.colsum = ctx->d_colsum; f.colelig = ctx->d_colelig; f.summ = a.summ;
  f.J = a.J; f.num_nodes = NN; f.nbatch = nbatch;
  f.gen = gen; f.first_cand = first_cand; f.key = a.key;
  f.list = ctx->d_collist; f.list_count = ctx->d_colcount;
  f.cur = a.cur; f.occ_count = ctx->d_occcount; f.occ_list = ctx->d_occlist;
  { TimedLaunch tl_(ctx, KK_COLS); colrepair_kernel<<<ctx->num_sms * 4, 128, 0, ctx->stream>>>(f); }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

RowsArgs base_rows_args(sched_ctx *ctx, const RngKey &key, const int32_t *d_k_cap, const uint8_t *d_active, int count) {
  RowsArgs a;
  const sched_config &c = ctx->cfg;
  a.cap = ctx->d_cap; a.k_cap = d_k_cap; a.active = d_active;
  a.rank = ctx->d_rank; a.order = ctx->d_order; a.dflag = ctx->d_dflag;
  a.P = c.population; a.J = c.num_jobs; a.num_nodes = c.num_nodes;
  a.k_max = c.k_max; a.n_max = c.n_max; a.num_elite = c.num_elite; a.count = count;
  a.thr = 0; a.gen = 0; a.first_cand = 0;
  a.key = key;
  a.src = nullptr; a.dst = nullptr; a.mode = ROWS_REPAIR; a.fitness_bits = nullptr;
  a.cur = nullptr; a.summ = nullptr; a.summ_in = nullptr;
  return a;
}

}  // namespace

int launch_repair(sched_ctx *ctx, RngKey key, const int32_t *d_k_cap, const uint8_t *d_active, int16_t *d_pop,
                  int32_t count, uint32_t first_candidate, uint32_t generation) {
  int rc = ensure_dflag(ctx, count);
  if (rc != SCHED_OK) return rc;
  RowsArgs a = base_rows_args(ctx, key, d_k_cap, d_active, count);
  a.mode = ROWS_REPAIR; a.src = d_pop; a.dst = d_pop;
  a.first_cand = first_candidate; a.gen = generation;
  return launch_rows_cols(ctx, a, d_pop, count, first_candidate, generation);
}

int launch_init_population(sched_ctx *ctx, RngKey key, const int32_t *d_k_cap, const uint8_t *d_active,
                           const int16_t *d_cur, int16_t *d_pop_out) {
  const int P = ctx->cfg.population;
  int rc = ensure_dflag(ctx, P);
  if (rc != SCHED_OK) return rc;
  RowsArgs a = base_rows_args(ctx, key, d_k_cap, d_active, P);
  a.mode = ROWS_INIT; a.src = d_cur; a.dst = d_pop_out;
  a.thr = ctx->cfg.thr_init; a.gen = GEN_INIT;
  a.cur = ctx->round_cur; a.summ = ctx->round_summ;
  return launch_rows_cols(ctx, a, d_pop_out, P, 0u, GEN_INIT);
}

// children first_child .. first_child + num_children - 1 (num_children < 0: all of them)
int launch_generation(sched_ctx *ctx, RngKey key, const int32_t *d_k_cap, const uint8_t *d_active,
                      const int16_t *d_pop_in, const float *d_fitness_in, int16_t *d_pop_out,
                      uint32_t generation, int first_child, int num_children) {
  const int P = num_children < 0 ? ctx->cfg.population : num_children;
  if (P == 0) return SCHED_OK;
  int rc = ensure_dflag(ctx, P);
  if (rc != SCHED_OK) return rc;
  RowsArgs a = base_rows_args(ctx, key, d_k_cap, d_active, P);
  a.first_cand = (uint32_t)first_child;
  a.mode = ROWS_GENERATION; a.src = d_pop_in; a.dst = d_pop_out;
  a.fitness_bits = (const uint32_t *)d_fitness_in;
  a.thr = ctx->cfg.thr_mutate; a.gen = generation;
  a.cur = ctx->round_cur; a.summ = ctx->round_summ; a.summ_in = ctx->round_summ_in;
  return launch_rows_cols(ctx, a, d_pop_out, P, (uint32_t)first_child, generation);
}

__global__ void set_round_kernel(uint32_t *dst, uint32_t value) { *dst = value; }

int launch_set_round(sched_ctx *ctx, uint32_t round) {
  set_round_kernel<<<1, 1, 0, ctx->stream>>>(ctx->d_round, round);
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

int launch_select_best(sched_ctx *ctx, const int16_t *d_pop, const float *d_fitness,
                       int16_t *d_best, float *d_best_fitness) {
  const int P = ctx->cfg.population;
  {
  TimedLaunch tl_(ctx, KK_BEST);
  best_index_kernel<<<1, 256, 0, ctx->stream>>>((const uint32_t *)d_fitness, P, ctx->d_best_idx,
                                                d_best_fitness);
  }
  SCHED_LAUNCH_CHECK(ctx);
  const size_t elems = (size_t)ctx->cfg.num_jobs * ctx->cfg.num_nodes;
  if (elems == 0 || !d_pop) return SCHED_OK;   // no dense population: the caller gathers the rows
  const int blocks = (int)((elems + 256 * 8 - 1) / (256 * 8));
  {
  TimedLaunch tl_(ctx, KK_COPY);
  copy_best_kernel<<<blocks > 1024 ? 1024 : blocks, 256, 0, ctx->stream>>>(d_pop, ctx->d_best_idx,
                                                                           elems, d_best);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}
