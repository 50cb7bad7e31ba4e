// A whole round's search in one launch (Sec. 4.3): initial population and generations by blocks that
// stay on the GPU and pass the population on through L2.
//
// A child needs little of the generation before it: the fitness of the four candidates its two
// tournaments drew and the rows of the two that won.  So the blocks do not meet between generations.  A
// candidate that is ready publishes its fitness key with the generation's tag; a child waits for the
// tags it needs (bounded; see wait_tag) and goes on, draws for the next generation being made while
// others are still busy.  Populations of four generations are kept in turn: a candidate may write over
// its rows of four generations ago once candidate 0, which waits for everybody in every generation, is two
// generations behind it.  The launch is cooperative, so that all blocks are on the GPU when one waits
// for another.
//
// A row is a 32-byte record: up to six occupied nodes (node << 16 | GPUs, ascending) and the row's term
// of the fitness sum (a row always serves the same job, so the term is fixed for the round).  A child copies
// the records of its parents' rows; only a row with more occupied nodes ("wide") also has contents.
// Rows of inactive jobs are left out.  One block works on one candidate at a time: a thread per row, a
// warp of its own for the perturbed rows, whose path is long and whose number is small.
// Operators, draws and the order of the fitness sums are those of the dense kernels: identical populations
// and fitness bits.
#include <algorithm>

#include "common.cuh"
#include "fitness_common.cuh"
#include "search_common.cuh"

namespace {

constexpr int REC_WORDS = 8;
constexpr int ENTRIES = 6;                      // occupied nodes a record holds
constexpr uint32_t NO_NODE = 0xFFFFFFFFu;       // an entry that is not used
constexpr uint32_t WIDE = 0xFFFFFFFEu;          // first entry of a row with more: its contents are elsewhere
constexpr int REC_TERM = 6;
constexpr int DEPTH = 4;                        // generations kept
constexpr int MAX_ROW_THREADS = 256;            // as the dense fitness kernel: the order of its sums
constexpr int STASH = 128;                      // perturbed rows whose draws are kept, further ones draw again
constexpr int SMEM_RECORDS = 256;              // up to this many jobs the child's records are kept in shared memory, too
constexpr int FLOW_MAX_JOBS = 8192, FLOW_MAX_NODES = 512;

__host__ __device__ inline int wide_stride(int NN) { return (NN + 7) & ~7; }

struct FlowRows {
  uint32_t *rec;             // [DEPTH][P][J][REC_WORDS]; rows of active jobs only, one behind the other
  int16_t *wide;             // [DEPTH][P][J][wide_stride] contents of wide rows
  uint32_t *cur_rec;         // [2][J][REC_WORDS] the current allocation after the row caps, and before them
  int16_t *cur_wide;         // [2][J][wide_stride]
  uint32_t *same;            // [J][REC_WORDS] entries of a row that equals the current allocation's (first one
                             // NO_NODE - 2: there is none with six nodes or fewer)
  float *pen;                // [J] penalty factor of a row that differs from the current allocation's
  uint16_t *act;             // [J] active jobs, ascending; act[J] .. : see num_act
  int *num_act;
  unsigned long long *pub;   // [DEPTH][P] tag << 32 | fitness key
  uint32_t *base;            // tag of the round's initial population
};
constexpr uint32_t NEVER = 0xFFFFFFFDu;

struct FlowArgs {
  FlowRows r;
  const int16_t *cap;        // [NN]
  const int32_t *k_cap;      // [J] or NULL
  const uint8_t *active;     // [J] or NULL
  const int16_t *cur;        // [J][NN] or NULL
  const float *age;          // [J]; read when the penalty is on
  const int32_t *restarts;
  const int16_t *rack;       // [NN] or NULL
  const float *table_rack;
  TermParams tp;             // tp.pen: r.pen when the penalty is on
  float delta;
  int P, J, NN, k_max, n_max, num_elite, generations, occ;
  int row_threads;           // then the warp of the perturbed rows, then the threads that draw (or none: the row threads do)
  uint32_t thr_init, thr_mutate;
  RngKey key;
  int rows_per_chunk, chunks;   // the dense fitness kernel's chunking, reproduced for identical sums
  float *fitness;            // [P]
  int16_t *best;             // [J][NN]
  float *best_fitness;
  unsigned int wait_limit;   // polls (a few hundred cycles each) before a wait gives up
  int *status;
};

__device__ __forceinline__ int entry_node(uint32_t e) { return (int)(e >> 16); }
__device__ __forceinline__ int entry_gpus(uint32_t e) { return (int)(e & 0xFFFFu); }

// One 32-byte record in one request, through L2: another block may have written it.
struct Record {
  uint32_t w[REC_WORDS];
};
__device__ __forceinline__ Record load_record(const uint32_t *p) {
  Record r;
  asm volatile("ld.global.cg.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
               : "l"(p) : "memory");
  return r;
}
__device__ __forceinline__ void store_record(uint32_t *p, const Record &r) {
  asm volatile("st.global.v8.u32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r.w[0]), "r"(r.w[1]), "r"(r.w[2]),
               "r"(r.w[3]), "r"(r.w[4]), "r"(r.w[5]), "r"(r.w[6]), "r"(r.w[7]) : "memory");
}

// ---- waiting and publishing --------------------------------------------------------------------
// The key published under `tag`; false when it has not come within the limit (the caller returns: the
// other blocks' waits run out the same way).  A thread that has waited calls waited() before the barrier
// behind which the block reads the rows, or before it publishes in its turn.
__device__ __noinline__ bool wait_tag(const unsigned long long *p, uint32_t tag, uint32_t &key, unsigned int limit, int *status) {
#pragma unroll 1
  for (unsigned int n = 0; n < limit; ++n) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    if ((uint32_t)(v >> 32) == tag) {
      key = (uint32_t)v;
      return true;
    }
  }
  atomicCAS(status, 0, SCHED_ERR_TIMEOUT);
  key = 0u;
  return false;
}
// Acquire: with the publisher's fence (release) and the block's barrier, what was written before the tag
// was published is seen by every thread of this block, and what was read before it lies behind it.  One
// fence after the polls that succeeded, not an acquire in each poll.  The one-way fence costs nothing that
// can be measured (testbed round 663 us with it and without, large 3.87 ms), fence.acq_rel, which also waits
// for this thread's own writes, 4 to 10 % (732 us, 4.03 ms).
__device__ __forceinline__ void waited() { asm volatile("fence.acquire.gpu;" ::: "memory"); }
__device__ __forceinline__ void publish(unsigned long long *p, uint32_t tag, uint32_t key) {
  const unsigned long long v = ((unsigned long long)tag << 32) | key;
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// ---- a row as its sorted list of occupied nodes, in registers -------------------------------------
constexpr int LIST = ENTRIES + 1;       // one more than a record holds: a perturbation may add before the caps take

__device__ __forceinline__ void list_totals(const uint32_t (&e)[LIST], int &K, int &N) {
  K = 0;
  N = 0;
#pragma unroll
  for (int k = 0; k < LIST; ++k) {
    const bool on = e[k] != NO_NODE;
    K += on ? entry_gpus(e[k]) : 0;
    N += on ? 1 : 0;
  }
}

// GPUs on a node, 0 when it is not occupied
__device__ __forceinline__ int list_at(const uint32_t (&e)[LIST], int node) {
  int v = 0;
#pragma unroll
  for (int k = 0; k < LIST; ++k) v = entry_node(e[k]) == node ? entry_gpus(e[k]) : v;
  return v;
}

// A[j][node] = v
__device__ __forceinline__ void list_set(uint32_t (&e)[LIST], int node, int v) {
  bool found = false;
#pragma unroll
  for (int k = 0; k < LIST; ++k)
    if (entry_node(e[k]) == node) {
      found = true;
      e[k] = v > 0 ? ((uint32_t)node << 16) | (uint32_t)v : NO_NODE;
    }
  uint32_t x = !found && v > 0 ? ((uint32_t)node << 16) | (uint32_t)v : NO_NODE;
#pragma unroll
  for (int k = 0; k < LIST; ++k) {      // a new entry to its place, a hole to the end
    const uint32_t lo = min(e[k], x);
    x = max(e[k], x);
    e[k] = lo;
  }
#pragma unroll
  for (int k = 0; k + 1 < LIST; ++k) {
    const uint32_t lo = min(e[k], e[k + 1]);
    e[k + 1] = max(e[k], e[k + 1]);
    e[k] = lo;
  }
}

// grow / shrink / relocate (Sec. 4.3), chosen by the row's draw
__device__ __forceinline__ void list_perturb(uint32_t (&e)[LIST], int N, uint32_t wy, uint32_t wz, uint32_t ww, int NN,
                                             const int16_t *s_cap) {
  const uint32_t op = bounded(wy, 3u);
  const int nd = (int)bounded(ww, (uint32_t)NN);
  int ns = -1, vs = 0;
  if (op != 0u && N > 0) {
    const int t = (int)bounded(wz, (uint32_t)N);
#pragma unroll
    for (int k = 0; k < LIST; ++k)
      if (k == t) { ns = entry_node(e[k]); vs = entry_gpus(e[k]); }
  }
  int node0 = -1, v0 = 0, node1 = -1;
  if (op == 0u) {
    node0 = nd;
    v0 = min(list_at(e, nd) + 1, (int)s_cap[nd]);
  } else if (ns >= 0) {
    if (op == 1u) {
      node0 = ns;
      v0 = vs - 1;
    } else if (nd != ns) {
      node0 = nd;
      v0 = min(list_at(e, nd) + vs, (int)s_cap[nd]);
      node1 = ns;
    }
  }
#pragma unroll 1
  for (int q = 0; q < 2; ++q) {
    const int node = q ? node1 : node0;
    if (node >= 0) list_set(e, node, q ? 0 : v0);
  }
}

// row caps: replicas above kc leave from the highest node index down, then occupied nodes beyond n_max
// are cleared from the highest index down
__device__ __forceinline__ void list_caps(uint32_t (&e)[LIST], int K, int kc, int n_max) {
  int excess = K - kc;
#pragma unroll
  for (int k = LIST - 1; k >= 0; --k) {
    if (e[k] != NO_NODE && excess > 0) {
      const int v = entry_gpus(e[k]), take = min(v, excess);
      excess -= take;
      e[k] = take == v ? NO_NODE : e[k] - (uint32_t)take;
    }
    if (k >= n_max) e[k] = NO_NODE;
  }
}

// ---- fitness terms ------------------------------------------------------------------------------
// table of a row by the racks its nodes lie in
__device__ __forceinline__ const float *table_of(const FlowArgs &a, int lo, int hi) { return lo < hi ? a.table_rack : a.tp.table; }

__device__ __forceinline__ const float *list_table(const FlowArgs &a, const uint32_t (&e)[LIST]) {
  if (!a.rack) return a.tp.table;
  int lo = 0x7fffffff, hi = -1;
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k)
    if (e[k] != NO_NODE && sched_index_ok(a.status, entry_node(e[k]) < a.NN, SCHED_CHK_NODE)) {
      const int r = (int)__ldg(a.rack + entry_node(e[k]));
      lo = min(lo, r);
      hi = max(hi, r);
    }
  return table_of(a, lo, hi);
}

// What a finished list's term needs from memory, asked for together (the table's entry, the job's penalty
// factor, the current allocation's entries), and the record it gives.
struct TermLoads {
  float speedup, pen;
  uint4 lo;
  uint2 hi;
};
__device__ __forceinline__ TermLoads list_loads(const FlowArgs &a, const uint32_t (&e)[LIST], int j, int K, int N) {
  TermLoads t;
  t.pen = 1.f;
  t.lo = make_uint4(0u, 0u, 0u, 0u);
  t.hi = make_uint2(0u, 0u);
  if (a.tp.pen) {
    t.lo = __ldg((const uint4 *)(a.r.same + (size_t)j * REC_WORDS));
    t.hi = __ldg((const uint2 *)(a.r.same + (size_t)j * REC_WORDS + 4));
    t.pen = __ldg(a.r.pen + j);
  }
  if (!sched_index_ok(a.status, j < a.J && K >= 0 && N >= 0 && N <= ENTRIES, SCHED_CHK_ENTRY)) K = N = 0;
  t.speedup = __ldg(list_table(a, e) + fitness_table_index(a.tp, j, K, N));
  return t;
}
__device__ __forceinline__ Record list_record(const FlowArgs &a, const uint32_t (&e)[LIST], const TermLoads &t) {
  const bool changed = t.lo.x != e[0] || t.lo.y != e[1] || t.lo.z != e[2] || t.lo.w != e[3] || t.hi.x != e[4] || t.hi.y != e[5];
  Record r;
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k) r.w[k] = e[k];
  r.w[REC_TERM] = __float_as_uint(fitness_term_with(a.tp, t.speedup, t.pen, changed));
  r.w[7] = 0u;
  return r;
}

// ---- rows laid out in shared memory, a warp each (wide rows, and lists that overflow) --------------
__device__ __forceinline__ void dense_from_list(int16_t *row, int NS, const Record &r, int lane, int *status) {
  for (int n = lane; n < NS; n += 32) row[n] = 0;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k)
    if (lane == k && r.w[k] != NO_NODE && sched_index_ok(status, entry_node(r.w[k]) < NS, SCHED_CHK_NODE))
      row[entry_node(r.w[k])] = (int16_t)entry_gpus(r.w[k]);
  __syncwarp();
}

__device__ __forceinline__ void dense_totals(const int16_t *row, int NN, int lane, int &K, int &N) {
  K = 0;
  N = 0;
#pragma unroll 1
  for (int n = lane; n < NN; n += 32) { K += row[n]; N += row[n] > 0; }
  K = __reduce_add_sync(0xffffffffu, K);
  N = __reduce_add_sync(0xffffffffu, N);
}

__device__ __forceinline__ void dense_caps(int16_t *row, int NN, int &K, int &N, int kc, int n_max, int lane) {
  if (K <= kc && N <= n_max) return;
  if (lane == 0) {
    int excess = K - kc;
#pragma unroll 1
    for (int n = NN - 1; n >= 0 && excess > 0; --n) {
      const int take = min((int)row[n], excess);
      row[n] = (int16_t)(row[n] - take);
      excess -= take;
    }
    int occ = 0;
#pragma unroll 1
    for (int n = 0; n < NN; ++n)
      if (row[n] > 0 && ++occ > n_max) row[n] = 0;
  }
  __syncwarp();
  dense_totals(row, NN, lane, K, N);
}

// the row as a record (and contents, when it is wide), with its term; all lanes return it
__device__ __noinline__ Record dense_record(const FlowArgs &a, const int16_t *row, int j, int K, int N, int16_t *wide, int lane) {
  const int NN = a.NN;
  int lo = 0x7fffffff, hi = -1, diff = 0, base = 0;
  uint32_t mine = NO_NODE;                // lane k: entry k
  const int16_t *cur = a.tp.pen ? a.cur + (size_t)j * NN : nullptr;
#pragma unroll 1
  for (int n0 = 0; n0 < NN; n0 += 32) {
    const int n = n0 + lane, v = n < NN ? (int)row[n] : 0;
    if (cur && n < NN) diff |= v != (int)cur[n];
    if (v > 0 && a.rack) {
      const int r = (int)__ldg(a.rack + n);
      lo = min(lo, r);
      hi = max(hi, r);
    }
    const unsigned m = __ballot_sync(0xffffffffu, v > 0);
    if (lane >= base && lane < base + __popc(m)) {
      const int at = (int)__fns(m, 0, lane - base + 1);
      mine = ((uint32_t)(n0 + at) << 16) | (uint32_t)row[n0 + at];
    }
    base += __popc(m);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  const bool changed = __any_sync(0xffffffffu, diff != 0);
  Record r;
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k) r.w[k] = __shfl_sync(0xffffffffu, mine, k);
  if (N > ENTRIES) {
    r.w[0] = WIDE;
#pragma unroll 1
    for (int n = lane; n < wide_stride(NN); n += 32) wide[n] = n < NN ? row[n] : (int16_t)0;
  }
  const float sp = __ldg(table_of(a, lo, hi) + fitness_table_index(a.tp, j, K, N));
  r.w[REC_TERM] = __float_as_uint(fitness_term_with(a.tp, sp, a.tp.pen ? a.r.pen[j] : 1.f, changed));
  r.w[7] = 0u;
  return r;
}

// ---------------------------------------------------------------------------------------
// Start of a round: the active jobs, and for each of them (a warp) the current allocation's row after the
// row caps (what an unperturbed row of the initial population is) and before them (what a perturbed one
// starts from), the list a row must equal to count as unchanged, and the penalty factor.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) flow_build_kernel(FlowArgs a) {
  __shared__ int16_t s_row[4][FLOW_MAX_NODES];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int J = a.J, NN = a.NN, NS = wide_stride(NN);
  if (blockIdx.x == 0 && warp == 0) {
    int n = 0;
#pragma unroll 1
    for (int j0 = 0; j0 < J; j0 += 32) {
      const bool on = j0 + lane < J && (!a.active || a.active[j0 + lane]);
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) a.r.act[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(j0 + lane);
      n += __popc(m);
    }
    if (lane == 0) *a.r.num_act = n;
  }
  int16_t *row = s_row[warp];
#pragma unroll 1
  for (int j = blockIdx.x * 4 + warp; j < J; j += gridDim.x * 4) {
    if (a.active && !a.active[j]) continue;
    long long raw = 0;
    bool in_range = true;
#pragma unroll 1
    for (int n = lane; n < NN; n += 32) {
      const int v = a.cur ? (int)a.cur[(size_t)j * NN + n] : 0;
      const int cl = min(max(v, 0), max((int)a.cap[n], 0));
      raw += v;
      in_range &= cl == v;
      row[n] = (int16_t)cl;
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) raw += __shfl_xor_sync(0xffffffffu, raw, off);
    in_range = __all_sync(0xffffffffu, in_range);
    if (a.tp.pen && lane == 0) a.r.pen[j] = raw > 0 ? realloc_factor(a.age[j], a.restarts[j], a.delta) : 1.f;
    __syncwarp();
    int K, N;
    dense_totals(row, NN, lane, K, N);
    const int kc = max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max));
#pragma unroll 1
    for (int caps = 1; caps >= 0; --caps) {     // before the caps (the second set), then after them (the first)
      if (!caps) dense_caps(row, NN, K, N, kc, a.n_max, lane);
      const size_t at = (size_t)caps * J + j;
      Record r = dense_record(a, row, j, K, N, a.r.cur_wide + at * NS, lane);
      if (lane == 0) store_record(a.r.cur_rec + at * REC_WORDS, r);
      if (caps && lane == 0) {
        if (!in_range || N > ENTRIES) r.w[0] = NEVER;
        store_record(a.r.same + (size_t)j * REC_WORDS, r);
      }
      __syncwarp();
    }
  }
}

// ---- shared memory of the generation kernel -----------------------------------------------------
struct FlowSmem {
  size_t act, term, info, node, occ, viol, cap, mut, mod, wide, slow, stash, flag, dense, rep, keys, sums, rec, total;
};

__host__ __device__ inline FlowSmem flow_smem(int P, int J, int NN, int occ, int warps, int chunks) {
  FlowSmem L;
  size_t off = 0;
#define TAKE(field, bytes) do { L.field = off; off += ((size_t)(bytes) + 15) & ~(size_t)15; } while (0)
  TAKE(act, (size_t)J * 2);
  TAKE(term, (size_t)J * 4);
  TAKE(info, (size_t)J);
  TAKE(node, (size_t)NN * 8);
  TAKE(occ, (size_t)NN * occ * 4);
  TAKE(viol, (size_t)NN);
  TAKE(cap, (size_t)NN * 2);
  TAKE(mut, 2 * (size_t)J * 2);
  TAKE(mod, (size_t)J * 2);
  TAKE(wide, (size_t)J * 2);
  TAKE(slow, (size_t)J * 2);
  TAKE(stash, 2 * (size_t)STASH * 16);
  TAKE(flag, 2 * (size_t)J);
  TAKE(dense, (size_t)warps * wide_stride(NN) * 2);
  TAKE(rep, 2 * (size_t)NN * 4);
  TAKE(keys, (size_t)P * 6);      // and a list of candidates behind them
  TAKE(sums, (size_t)chunks * 8 * 8);
  TAKE(rec, J <= SMEM_RECORDS ? (size_t)J * REC_WORDS * 4 : 0);
#undef TAKE
  L.total = off;
  return L;
}

constexpr int INFO_DIST = 1;        // the row spanned two nodes or more after the row pass (interference snapshot)
constexpr int INFO_CHANGED = 2;     // a node's decision changes it
constexpr int INFO_WIDE = 4;

// Block-wide minimum and exclusive prefix sum (s_red: a word per warp); both end with a barrier.
__device__ __noinline__ int block_min(int v, int *s_red, int nwarps) {
  v = __reduce_min_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = s_red[0];
#pragma unroll 1
  for (int w = 1; w < nwarps; ++w) r = min(r, s_red[w]);
  __syncthreads();
  return r;
}
__device__ __noinline__ int block_exscan(int v, int *s_red, int nwarps, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += u;
  }
  if (lane == 31) s_red[warp] = incl;
  __syncthreads();
  int before = 0;
  total = 0;
#pragma unroll 1
  for (int w = 0; w < nwarps; ++w) {
    const int t = s_red[w];
    if (w < warp) before += t;
    total += t;
  }
  __syncthreads();
  return before + incl - v;
}

// GPUs of a finished row of this block's candidate on a node
__device__ __noinline__ int row_at(const uint32_t *rec, const int16_t *wide, int NS, int jc, int node) {
  const Record r = load_record(rec + (size_t)jc * REC_WORDS);
  if (r.w[0] == WIDE) return (int)__ldcg(wide + (size_t)jc * NS + node);
  int v = 0;
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k) v = entry_node(r.w[k]) == node ? entry_gpus(r.w[k]) : v;
  return v;
}

// everything a block knows about the candidate it is working on
struct Work {
  const uint32_t *src_a, *src_b;      // parents' records (initial population: the current allocation after and before the caps)
  const int16_t *wide_a, *wide_b;     // and contents
  uint32_t *rec;                      // the child's
  int16_t *wide;
  uint32_t c, gen, round;
  bool init;
};

// An elite child: the records (and contents) of the candidate of its rank, as they are.
__device__ __noinline__ void copy_candidate(const FlowArgs &a, const uint32_t *from, const int16_t *wide_from, uint32_t *to,
                                            int16_t *wide_to, int rows) {
  const int NS = wide_stride(a.NN);
#pragma unroll 4
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    const Record r = load_record(from + (size_t)i * REC_WORDS);
    store_record(to + (size_t)i * REC_WORDS, r);
    if (r.w[0] == WIDE) {
#pragma unroll 1
      for (int v = 0; v < NS / 8; ++v)
        ((uint4 *)(wide_to + (size_t)i * NS))[v] = __ldcg((const uint4 *)(wide_from + (size_t)i * NS) + v);
    }
  }
}

__global__ void __launch_bounds__(2 * MAX_ROW_THREADS + 32, 2) flow_kernel(const __grid_constant__ FlowArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int J = a.J, NN = a.NN, NS = wide_stride(NN), P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5, T = a.row_threads;
  const int draw_t = (int)blockDim.x > T + 32 ? tid - (T + 32) : tid < T ? tid : -1;    // place among the drawing threads
  const FlowSmem L = flow_smem(P, J, NN, a.occ, nwarps, a.chunks);
  uint16_t *s_act = (uint16_t *)(smem + L.act);
  float *s_term = (float *)(smem + L.term);                   // by job, 0 where there is none
  uint8_t *s_info = smem + L.info;                            // by row
  int *s_tot = (int *)(smem + L.node);                        // GPUs placed on the node
  uint32_t *s_cnt = (uint32_t *)(s_tot + NN);                 // distributed jobs on it | occupants << 16
  uint32_t *s_occ = (uint32_t *)(smem + L.occ);               // row | GPUs << 13 | place in the record (7: wide) << 25 | distributed << 31
  uint8_t *s_viol = smem + L.viol;                            // the node's column is to be walked
  int16_t *s_cap = (int16_t *)(smem + L.cap);
  uint16_t *s_mut2 = (uint16_t *)(smem + L.mut), *s_mod = (uint16_t *)(smem + L.mod);
  uint16_t *s_wide = (uint16_t *)(smem + L.wide), *s_slow = (uint16_t *)(smem + L.slow);
  uint4 *s_stash2 = (uint4 *)(smem + L.stash);
  uint8_t *s_flag2 = smem + L.flag;                          // by row: 1 from the second parent, 2 perturbed
  uint32_t *s_rec = J <= SMEM_RECORDS ? (uint32_t *)(smem + L.rec) : nullptr;
  int16_t *s_dense = (int16_t *)(smem + L.dense) + (size_t)warp * NS;
  uint32_t *s_rep2 = (uint32_t *)(smem + L.rep);
  uint32_t *s_keys = (uint32_t *)(smem + L.keys);
  double *s_sums = (double *)(smem + L.sums);
  __shared__ int s_nmut2[2], s_nwide, s_nslow, s_nmod, s_walk, s_ok, s_po;
  __shared__ uint32_t s_par[2], s_sel[2][4];
  __shared__ int s_red[2 * MAX_ROW_THREADS / 32 + 1];

  const uint32_t round = __ldg(a.key.round_ptr), base = __ldg(a.r.base);
  const int JA = *a.r.num_act;
#pragma unroll 1
  for (int i = tid; i < JA; i += blockDim.x) s_act[i] = a.r.act[i];
#pragma unroll 1
  for (int i = tid; i < J; i += blockDim.x) s_term[i] = 0.f;
#pragma unroll 1
  for (int i = tid; i < a.chunks * 8; i += blockDim.x) s_sums[i] = 0.0;
#pragma unroll 1
  for (int i = tid; i < NN; i += blockDim.x) { s_cap[i] = (int16_t)max((int)a.cap[i], 0); s_tot[i] = 0; s_cnt[i] = 0u; s_viol[i] = 0; }
  if (tid == 0) { s_nmut2[0] = s_nmut2[1] = 0; s_nwide = 0; s_nslow = 0; s_nmod = 0; s_walk = 0; s_ok = 1; }
  __syncthreads();
  const bool rep_ahead = J <= SMEM_RECORDS;       // the nodes' repair numbers are drawn ahead, too
  const size_t cand_rec = (size_t)J * REC_WORDS, cand_wide = (size_t)J * NS;
  auto rec_of = [&](int step, uint32_t c) { return a.r.rec + ((size_t)(step & (DEPTH - 1)) * P + c) * cand_rec; };
  auto wide_of = [&](int step, uint32_t c) { return a.r.wide + ((size_t)(step & (DEPTH - 1)) * P + c) * cand_wide; };
  auto pub_of = [&](int step, uint32_t c) { return a.r.pub + (size_t)(step & (DEPTH - 1)) * P + c; };

  // A candidate's random numbers of a step: each row's parent and whether it is perturbed, the perturbed
  // rows' list.  Nothing in it waits for another block, so it is done a step ahead - by threads of their
  // own where the GPU has room for them, else by the row threads while the perturbed rows are worked on.
  // Two sets.
  auto draw_step = [&](int s, uint32_t c, int set) {
    const bool init = s == 0;
    const uint32_t gen = (uint32_t)(s - 1);                 // (GEN_INIT is -1)
    if (!init && (int)c < a.num_elite) return;
    uint16_t *s_mut = s_mut2 + set * J;
    uint8_t *s_flag = s_flag2 + set * J;
#pragma unroll 1
    for (int jc = draw_t; jc < JA; jc += T) {
      const uint32_t j = s_act[jc];
      u32x4 m;
      uint32_t x = 0u;
      draw_two(a.key.k0, round, j, c, gen, SLOT_XOVER, init ? SLOT_INIT : SLOT_MUTATE, x, m);
      const bool sec = !init && (x >> 31) != 0u, mut = init ? c > 0u && m.x < a.thr_init : m.x < a.thr_mutate;
      s_flag[jc] = (sec ? 1 : 0) | (mut ? 2 : 0);
      if (mut) {
        const int i = atomicAdd(&s_nmut2[set], 1);
        if (!sched_index_ok(a.status, i < J, SCHED_CHK_LIST)) continue;
        s_mut[i] = (uint16_t)(jc | (sec ? 0x8000 : 0));
        if (i < STASH) s_stash2[set * STASH + i] = make_uint4(m.y, m.z, m.w, (uint32_t)max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max)));
      }
    }
    if (rep_ahead) {
#pragma unroll 1
      for (int n = T - 1 - draw_t; n < NN; n += T) {
        uint32_t x;
        u32x4 y;
        draw_two(a.key.k0, round, (uint32_t)n, c, gen, SLOT_REPAIR_INTF, SLOT_REPAIR_CAP, x, y);
        s_rep2[set * NN + n] = bounded(x, (uint32_t)J) | (bounded(y.x, (uint32_t)J) << 16);
      }
    }
    if (draw_t < 32 && !init) {
      const u32x4 sel = draw_one(a.key.k0, round, 0u, c, gen, SLOT_SELECT);
      if (lane < 4) s_sel[set][lane] = bounded(lane == 0 ? sel.x : lane == 1 ? sel.y : lane == 2 ? sel.z : sel.w, (uint32_t)P);
    }
  };
  // Items: this block's candidates of step 0 (the initial population), of step 1 (generation 0), ...; the
  // item before the first only draws.
  int s_at = 0, item = -1;
  uint32_t c_at = blockIdx.x;
#pragma unroll 1
  while (s_at <= a.generations) {
      int s = s_at;
      uint32_t c = c_at;
      asm volatile("" : "+r"(s));               // (one copy of the code for all steps)
      if (item >= 0) {
        c_at += gridDim.x;
        if (c_at >= (uint32_t)P) { c_at = blockIdx.x; ++s_at; }
      }
      Work w;
      w.c = c; w.init = s == 0; w.gen = w.init ? GEN_INIT : (uint32_t)(s - 1); w.round = round;
      w.rec = rec_of(s, c); w.wide = wide_of(s, c);
      const bool elite = item >= 0 && !w.init && (int)c < a.num_elite;

      const int set = item & 1;
      uint16_t *const s_mut = s_mut2 + set * J;
      const uint8_t *const s_flag = s_flag2 + set * J;
      uint4 *const s_stash = s_stash2 + set * STASH;
      uint32_t *const s_rep = s_rep2 + set * NN;
      // ---- parents ----------------------------------------------------------------------------------
      // The candidate of its rank for an elite child (which needs every key), else the better-ranked of
      // two random pairs (which needs four).  Candidate 0 waits for every key in any case: that it has
      // published step t tells everybody that nobody reads step t - 2 any more.
      if (item >= 0 && !w.init) {
        if (elite || c == 0u) {
          bool ok = true;
#pragma unroll 1
          for (int i = tid; i < P && ok; i += blockDim.x) {
            uint32_t k;
            ok = wait_tag(pub_of(s - 1, i), base + (uint32_t)(s - 1), k, a.wait_limit, a.status);
            s_keys[i] = k;
          }
          waited();
          if (!ok) s_ok = 0;
          __syncthreads();
          if (elite && warp == 0 && s_ok) {
            const int i = candidate_of_rank(s_keys, P, (int)c, (uint16_t *)(s_keys + P), lane);
            if (lane == 0) s_par[0] = s_par[1] = (uint32_t)i;
          }
        }
        if (warp == T / 32) {
          uint32_t k = 0u;
          bool ok = true;
          const uint32_t mine = s_sel[set][lane & 3];
          if (lane < 4 && !elite) ok = wait_tag(pub_of(s - 1, mine), base + (uint32_t)(s - 1), k, a.wait_limit, a.status);
          if (lane == 4 && s >= DEPTH) ok = wait_tag(pub_of(s - 2, 0u), base + (uint32_t)(s - 2), k, a.wait_limit, a.status);
          waited();
          if (!__all_sync(0xffffffffu, ok) && lane == 0) s_ok = 0;
          const uint32_t other = __shfl_down_sync(0xffffffffu, mine, 1), ko = __shfl_down_sync(0xffffffffu, k, 1);
          if (!elite && (lane == 0 || lane == 2)) s_par[lane >> 1] = (uint32_t)tournament_winner(k, (int)mine, ko, (int)other);
        }
      }
      __syncthreads();
      if (!s_ok) return;                        // (a wait ran out: the status says so)
      if (!sched_index_ok(a.status, w.init || (s_par[0] < (uint32_t)P && s_par[1] < (uint32_t)P), SCHED_CHK_SLOT)) return;
      const uint32_t elite_key = elite ? s_keys[s_par[0]] : 0u;
      // (initial population: an unperturbed row is the current allocation's after the row caps, a perturbed one
      // starts from it before them; rows of the current allocation lie by job)
      w.src_a = w.init ? a.r.cur_rec : rec_of(s - 1, s_par[0]);
      w.wide_a = w.init ? a.r.cur_wide : wide_of(s - 1, s_par[0]);
      w.src_b = w.init ? a.r.cur_rec + cand_rec : rec_of(s - 1, s_par[1]);
      w.wide_b = w.init ? a.r.cur_wide + cand_wide : wide_of(s - 1, s_par[1]);

      // a row's occupants into the nodes' totals and lists
      auto add_occupant = [&](int jc, int k_rec, uint32_t e, uint32_t dist) {
        const int n = entry_node(e);
        if (!sched_index_ok(a.status, n < NN && jc < JA && entry_gpus(e) <= 2047, SCHED_CHK_NODE)) return;
        atomicAdd(&s_tot[n], entry_gpus(e));
        const uint32_t k = atomicAdd(&s_cnt[n], (dist ? 1u : 0u) | (1u << 16)) >> 16;
        if (k < (uint32_t)a.occ) s_occ[n * a.occ + k] = (uint32_t)jc | ((uint32_t)entry_gpus(e) << 13) | ((uint32_t)k_rec << 25) | dist;
      };
      // small problems find a row of their own child again in shared memory
      auto keep_record = [&](int jc, const Record &r) {
        if (!s_rec) return;
        ((uint4 *)(s_rec + jc * REC_WORDS))[0] = make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]);
        ((uint4 *)(s_rec + jc * REC_WORDS))[1] = make_uint4(r.w[4], r.w[5], r.w[6], r.w[7]);
      };
      auto own_record = [&](int jc) {
        if (!s_rec) return load_record(w.rec + (size_t)jc * REC_WORDS);
        const uint4 x = ((const uint4 *)(s_rec + jc * REC_WORDS))[0], y = ((const uint4 *)(s_rec + jc * REC_WORDS))[1];
        return Record{{x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w}};
      };
      const int nmut = item >= 0 ? s_nmut2[set] : 0;
      if (elite) {
        copy_candidate(a, w.src_a, w.wide_a, w.rec, w.wide, JA);
      } else if (tid < T && item >= 0) {
        // ---- unperturbed rows, a thread each; four at a time, so that their loads travel together ------
        constexpr int RB = 4;
#pragma unroll 1
        for (int jc0 = tid; jc0 < JA; jc0 += RB * T) {
          Record rec[RB];
          uint32_t flag[RB];
#pragma unroll
          for (int q = 0; q < RB; ++q) {
            const int jc = min(jc0 + q * T, JA - 1);
            flag[q] = jc0 + q * T < JA ? s_flag[jc] : 2u;
            const uint32_t *src = (flag[q] & 1u) ? w.src_b : w.src_a;
            rec[q] = load_record(src + (size_t)(w.init ? (int)s_act[jc] : jc) * REC_WORDS);
          }
#pragma unroll
          for (int q = 0; q < RB; ++q) {
            const int jc = jc0 + q * T;
            if (flag[q] & 2u) continue;
            store_record(w.rec + (size_t)jc * REC_WORDS, rec[q]);
            keep_record(jc, rec[q]);
            s_term[s_act[jc]] = __uint_as_float(rec[q].w[REC_TERM]);
            if (rec[q].w[0] == WIDE) {
              s_info[jc] = INFO_DIST | INFO_WIDE;
              const int at = atomicAdd(&s_nwide, 1);
              if (sched_index_ok(a.status, at < J, SCHED_CHK_LIST)) s_wide[at] = (uint16_t)(jc | ((flag[q] & 1u) ? 0x8000 : 0));
              continue;
            }
            const uint32_t dist = rec[q].w[1] != NO_NODE ? 0x80000000u : 0u;
            s_info[jc] = dist ? INFO_DIST : 0;
            if (rec[q].w[0] != NO_NODE) add_occupant(jc, 0, rec[q].w[0], dist);
#pragma unroll 1
            for (int k = 1; k < ENTRIES; ++k) {           // (few rows have more: one copy of the code)
              uint32_t e = rec[q].w[1];
#pragma unroll
              for (int z = 2; z < ENTRIES; ++z) e = z == k ? rec[q].w[z] : e;
              if (e == NO_NODE) break;
              add_occupant(jc, k, e, dist);
            }
          }
        }
      }
      if (draw_t >= 0) {
        if (s_at <= a.generations) draw_step(s_at, c_at, set ^ 1);
      } else if (tid >= T && !elite) {
        // ---- perturbed rows: the last warp, a lane each --------------------------------------------------
#pragma unroll 1
        for (int i = lane; i < nmut; i += 32) {
          const int jc = s_mut[i] & 0x7FFF;
          if (!sched_index_ok(a.status, i < J && jc < JA, SCHED_CHK_LIST)) continue;
          const int j = s_act[jc];
          const uint32_t *src = (w.init || (s_mut[i] >> 15)) ? w.src_b : w.src_a;
          const Record rec = load_record(src + (size_t)(w.init ? j : jc) * REC_WORDS);
          uint4 st;
          if (i < STASH) {
            st = s_stash[i];
          } else {
            const u32x4 m = draw_one(a.key.k0, round, (uint32_t)j, c, w.gen, w.init ? SLOT_INIT : SLOT_MUTATE);
            st = make_uint4(m.y, m.z, m.w, (uint32_t)max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max)));
          }
          bool slow = rec.w[0] == WIDE;
          if (!slow) {
            uint32_t e[LIST];
#pragma unroll
            for (int k = 0; k < ENTRIES; ++k) e[k] = rec.w[k];
            e[ENTRIES] = NO_NODE;
            int K, N;
            list_totals(e, K, N);
            list_perturb(e, N, st.x, st.y, st.z, NN, s_cap);
            list_totals(e, K, N);
            if (K > (int)st.w || N > a.n_max) {
              list_caps(e, K, (int)st.w, a.n_max);
              list_totals(e, K, N);
            }
            slow = e[ENTRIES] != NO_NODE;
            if (!slow) {
              const uint32_t dist = N >= 2 ? 0x80000000u : 0u;
              const TermLoads loads = list_loads(a, e, j, K, N);     // (on their way while the nodes are added up)
              s_info[jc] = dist ? INFO_DIST : 0;
#pragma unroll 1
              for (int k = 0; k < N; ++k) {
                uint32_t x = e[0];
#pragma unroll
                for (int z = 1; z < ENTRIES; ++z) x = z == k ? e[z] : x;
                add_occupant(jc, k, x, dist);
              }
              const Record out = list_record(a, e, loads);
              store_record(w.rec + (size_t)jc * REC_WORDS, out);
              keep_record(jc, out);
              s_term[j] = __uint_as_float(out.w[REC_TERM]);
            }
          }
          if (slow) {
            const int at = atomicAdd(&s_nslow, 1);
            if (sched_index_ok(a.status, at < J, SCHED_CHK_LIST)) s_slow[at] = s_mut[i];
          }
        }
      }
      __syncthreads();
      if (elite || item < 0) {
        if (elite && tid == 0) {
          publish(pub_of(s, c), base + (uint32_t)s, elite_key);
          if (s == a.generations) a.fitness[c] = __uint_as_float(elite_key ^ ((elite_key >> 31) ? 0x80000000u : 0xFFFFFFFFu));
        }
        ++item;
        continue;
      }

      // ---- wide rows, a warp each -------------------------------------------------------------------
      if (s_nwide | s_nslow) {
#pragma unroll 1
        for (int i = warp; i < s_nwide + s_nslow; i += nwarps) {
          const bool slow = i >= s_nwide;
          const int x = slow ? s_slow[i - s_nwide] : s_wide[i], jc = x & 0x7FFF;
          if (!sched_index_ok(a.status, jc < JA, SCHED_CHK_LIST)) continue;
          const int j = s_act[jc];
          const bool sec = (x >> 15) || (w.init && slow);
          const int at = w.init ? j : jc;
          const Record rec = load_record((sec ? w.src_b : w.src_a) + (size_t)at * REC_WORDS);
          if (rec.w[0] == WIDE) {
            const int16_t *from = (sec ? w.wide_b : w.wide_a) + (size_t)at * NS;
#pragma unroll 1
            for (int n = lane; n < NS; n += 32) {
              const int16_t v = __ldcg(from + n);
              s_dense[n] = v;
              if (!slow) w.wide[(size_t)jc * NS + n] = v;
            }
            __syncwarp();
          } else {
            dense_from_list(s_dense, NS, rec, lane, a.status);
          }
          if (slow) {
            int K, N;
            dense_totals(s_dense, NN, lane, K, N);
            const u32x4 m = draw_one(a.key.k0, round, (uint32_t)j, c, w.gen, w.init ? SLOT_INIT : SLOT_MUTATE);
            const uint32_t op = bounded(m.y, 3u);
            const int nd = (int)bounded(m.w, (uint32_t)NN);
            if (op == 0u) {
              if (lane == 0) s_dense[nd] = (int16_t)min((int)s_dense[nd] + 1, (int)s_cap[nd]);
            } else if (N > 0) {
              int ns = nth_occupied(s_dense, NN, bounded(m.z, (uint32_t)N), lane);
              if (!sched_index_ok(a.status, ns >= 0 && ns < NN && nd < NN, SCHED_CHK_NODE)) ns = nd;
              if (lane == 0 && op == 1u) s_dense[ns] = (int16_t)(s_dense[ns] - 1);
              if (lane == 0 && op == 2u && nd != ns) {
                s_dense[nd] = (int16_t)min((int)s_dense[nd] + (int)s_dense[ns], (int)s_cap[nd]);
                s_dense[ns] = 0;
              }
            }
            __syncwarp();
            dense_totals(s_dense, NN, lane, K, N);
            dense_caps(s_dense, NN, K, N, max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max)), a.n_max, lane);
            const Record out = dense_record(a, s_dense, j, K, N, w.wide + (size_t)jc * NS, lane);
            if (lane == 0) {
              store_record(w.rec + (size_t)jc * REC_WORDS, out);
              keep_record(jc, out);
              s_term[j] = __uint_as_float(out.w[REC_TERM]);
              s_info[jc] = (N >= 2 ? INFO_DIST : 0) | (N > ENTRIES ? INFO_WIDE : 0);
            }
            __syncwarp();
          }
          const uint32_t dist = (s_info[jc] & INFO_DIST) ? 0x80000000u : 0u;
          const bool wide = (s_info[jc] & INFO_WIDE) != 0;
          int before = 0;
#pragma unroll 1
          for (int n0 = 0; n0 < NN; n0 += 32) {
            const int n = n0 + lane, v = n < NN ? (int)s_dense[n] : 0;
            const unsigned m = __ballot_sync(0xffffffffu, v > 0);
            const int k = before + __popc(m & ((1u << lane) - 1u));
            if (v > 0) add_occupant(jc, wide ? 7 : k, ((uint32_t)n << 16) | (uint32_t)v, dist);
            before += __popc(m);
          }
          __syncwarp();
        }
        __syncthreads();
      }

      // A decision goes straight into the row: entry k of its record (0 GPUs: taken out when the row is
      // finished), or its contents.  Decisions of different nodes touch different words.
      auto set_entry = [&](int jc, int k, int n, int v) {
        if (!sched_index_ok(a.status, jc < JA && n < NN && (k == 7 || k < ENTRIES), SCHED_CHK_ENTRY)) return;
        if (k == 7) w.wide[(size_t)jc * NS + n] = (int16_t)v;
        else if (s_rec) s_rec[jc * REC_WORDS + k] = ((uint32_t)n << 16) | (uint32_t)v;
        else w.rec[(size_t)jc * REC_WORDS + k] = ((uint32_t)n << 16) | (uint32_t)v;
      };

      // ---- node decisions: a lane looks at a node, groups of 16 lanes decide the nodes that hold two
      // distributed jobs or more GPUs than they have; nodes are dealt out round robin, so that violations
      // spread over the warps ---------------------------------------------------------------------------
#pragma unroll 1
      for (int n0 = warp; n0 < NN; n0 += 32 * nwarps) {
        const int n_l = n0 + lane * nwarps;
        bool bad = false;
        if (n_l < NN) bad = (s_cnt[n_l] & 0xFFFFu) >= 2u || s_tot[n_l] > (int)s_cap[n_l];
        unsigned todo = __ballot_sync(0xffffffffu, bad);
        if (todo == 0u) continue;
        uint32_t rep_l = 0u;                    // the two rotation offsets, below 8192 each
        if (bad) {
          if (rep_ahead) {
            rep_l = s_rep[n_l];
          } else {
            uint32_t x;
            u32x4 y;
            draw_two(a.key.k0, round, (uint32_t)n_l, c, w.gen, SLOT_REPAIR_INTF, SLOT_REPAIR_CAP, x, y);
            rep_l = bounded(x, (uint32_t)J) | (bounded(y.x, (uint32_t)J) << 16);
            s_rep[n_l] = rep_l;                 // (a walked column wants it again)
          }
        }
        __syncwarp();
#pragma unroll 1
        while (todo) {
          const int b0 = __ffs(todo) - 1;
          todo &= todo - 1;
          int b1 = -1;
          if (todo) { b1 = __ffs(todo) - 1; todo &= todo - 1; }
          const int b = (lane & 16) ? b1 : b0, sub = lane & 15;
          const uint32_t rep = __shfl_sync(0xffffffffu, rep_l, max(b, 0));
          const int n = n0 + max(b, 0) * nwarps, count = b >= 0 ? (int)(s_cnt[n] >> 16) : 0;
          const bool listed = count <= a.occ, have = listed && sub < count;   // else: walked below
          const uint32_t e = have ? s_occ[n * a.occ + sub] : 0u;
          const int jc = (int)(e & 0x1FFFu);
          const int j = have && sched_index_ok(a.status, jc < JA, SCHED_CHK_LIST) ? (int)s_act[jc] : 0;
          int ri = j - (int)(rep & 0xFFFFu), rc = have ? j - (int)(rep >> 16) : 0x3fffffff;
          if (ri < 0) ri += J;
          if (rc < 0) rc += J;
          const int most = max(__shfl_sync(0xffffffffu, count, 0), __shfl_sync(0xffffffffu, count, 16));
          const int v = decide(have ? (int)((e >> 13) & 0x7FFu) : 0, (e >> 31) != 0u, have, min(most, a.occ), (s_cnt[n] & 0xFFFFu) >= 2u, s_tot[n], (int)s_cap[n], ri, rc);
          const bool changed = have && v != (int)((e >> 13) & 0x7FFu);
          if (changed) {
            set_entry(jc, (int)((e >> 25) & 7u), n, v);
            // (bytes, so the word around it is updated as a whole)
            const uint32_t bit = (uint32_t)INFO_CHANGED << (8 * (jc & 3));
            if (sched_index_ok(a.status, jc < JA, SCHED_CHK_LIST) && (atomicOr((uint32_t *)s_info + (jc >> 2), bit) & bit) == 0u) {
              const int at = atomicAdd(&s_nmod, 1);
              if (sched_index_ok(a.status, at < J, SCHED_CHK_LIST)) s_mod[at] = (uint16_t)jc;
            }
          }
          if (b >= 0 && sub == 0 && !listed) { s_viol[n] = 1; s_walk = 1; }
          __syncwarp();
        }
      }
      __syncthreads();

      // ---- rows the decisions change ------------------------------------------------------------------
      // a row without the entries that were taken out, and its new term; by one thread (records), one warp (wide)
      auto finish_row = [&](int jc) {
        const int j = s_act[jc];
        const Record rec = own_record(jc);
        uint32_t e[LIST];
        int holes = 0;
#pragma unroll
        for (int k = 0; k < ENTRIES; ++k) {
          const bool out = entry_gpus(rec.w[k]) == 0;       // (an unused entry is not: its low half is all ones)
          e[k] = out ? NO_NODE : rec.w[k];
          holes += out ? 1 : 0;
        }
        e[ENTRIES] = NO_NODE;
#pragma unroll 1
        for (int h = 0; h < holes; ++h) {
#pragma unroll
          for (int k = 0; k + 1 < ENTRIES; ++k) {           // the last hole to the end
            const uint32_t lo = min(e[k], e[k + 1]);
            e[k + 1] = max(e[k], e[k + 1]);
            e[k] = lo;
          }
        }
        int K, N;
        list_totals(e, K, N);
        const Record out = list_record(a, e, list_loads(a, e, j, K, N));
        store_record(w.rec + (size_t)jc * REC_WORDS, out);
        keep_record(jc, out);
        s_term[j] = __uint_as_float(out.w[REC_TERM]);
      };
      auto finish_wide = [&](int jc) {
        int16_t *row = w.wide + (size_t)jc * NS;
#pragma unroll 1
        for (int n = lane; n < NN; n += 32) s_dense[n] = __ldcg(row + n);
        __syncwarp();
        int K, N;
        dense_totals(s_dense, NN, lane, K, N);
        const Record out = dense_record(a, s_dense, s_act[jc], K, N, row, lane);
        if (lane == 0) {
          store_record(w.rec + (size_t)jc * REC_WORDS, out);
          keep_record(jc, out);
          s_term[s_act[jc]] = __uint_as_float(out.w[REC_TERM]);
          if (N <= ENTRIES) s_info[jc] &= ~INFO_WIDE;
        }
        __syncwarp();
      };
      const int nmod = s_nmod;
#pragma unroll 1
      for (int i = tid; i < nmod; i += blockDim.x) {
        const int jc = s_mod[i];
        if (!(s_info[jc] & INFO_WIDE)) finish_row(jc);
      }
      if (s_nwide | s_nslow) {                  // wide rows among them
        __syncthreads();                        // (one may turn into a record here: not to be taken for one above)
#pragma unroll 1
        for (int i = warp; i < nmod; i += nwarps) {
          const int jc = s_mod[i];
          if (s_info[jc] & INFO_WIDE) finish_wide(jc);
        }
      }

      // ---- nodes with more occupants than a list holds: the block walks the column, node by node ------
      // Thread t looks after the consecutive rows [t * rpt, (t + 1) * rpt).  Interference: the first
      // distributed occupant in rotated job order stays.  Capacity: a block-wide prefix sum in job order gives
      // every row the GPUs that come before it in rotated order.
      if (s_walk) {
        __syncthreads();
        const int rpt = (JA + (int)blockDim.x - 1) / (int)blockDim.x;
        const int lo = min(JA, tid * rpt), hi = min(JA, lo + rpt);
#pragma unroll 1
        for (int n = 0; n < NN; ++n) {
          if (!s_viol[n]) continue;
          const uint32_t rep = s_rep[n];
          const bool intf = (s_cnt[n] & 0xFFFFu) >= 2u;
          auto dist = [&](int jc) { return (s_info[jc] & INFO_DIST) != 0; };
          int keep = -1;
          if (intf) {
            int best = 0x7fffffff;
#pragma unroll 1
            for (int jc = lo; jc < hi; ++jc)
              if (dist(jc) && row_at(w.rec, w.wide, NS, jc, n) > 0) {
                int t = (int)s_act[jc] - (int)(rep & 0xFFFFu);
                if (t < 0) t += J;
                best = min(best, t);
              }
            keep = (int)(rep & 0xFFFFu) + block_min(best, s_red, nwarps);     // the job that stays
            if (keep >= J) keep -= J;
          }
          auto stays = [&](int jc) {
            const int v = row_at(w.rec, w.wide, NS, jc, n);
            return intf && dist(jc) && v > 0 && (int)s_act[jc] != keep ? 0 : v;
          };
          int mine = 0, total;
#pragma unroll 1
          for (int jc = lo; jc < hi; ++jc) mine += stays(jc);
          int running = block_exscan(mine, s_red, nwarps, total);
          const int excess = total - (int)s_cap[n], o = (int)(rep >> 16);
          int p_o = 0;                          // GPUs of the rows before the offset in job order
          if (excess > 0) {
            if (tid == 0) s_po = total;         // (no active job at or behind the offset)
            __syncthreads();
            int p = running;
#pragma unroll 1
            for (int jc = lo; jc < hi; ++jc) {
              if ((int)s_act[jc] >= o && (jc == 0 || (int)s_act[jc - 1] < o)) s_po = p;
              p += stays(jc);
            }
            __syncthreads();
            p_o = s_po;
          }
#pragma unroll 1
          for (int jc = lo; jc < hi; ++jc) {
            const int v = row_at(w.rec, w.wide, NS, jc, n), v_eff = stays(jc);
            int take = 0;
            if (excess > 0) {
              const int ahead = (int)s_act[jc] >= o ? running - p_o : total - p_o + running;
              take = min(v_eff, max(excess - ahead, 0));
            }
            running += v_eff;
            s_mod[jc] = v_eff - take == v ? 0 : 1;
            if (v_eff - take != v) {            // into the row
              int k = 7;
              if (!(s_info[jc] & INFO_WIDE)) {
                const Record rec = own_record(jc);
#pragma unroll
                for (int z = 0; z < ENTRIES; ++z) k = entry_node(rec.w[z]) == n ? z : k;
              }
              set_entry(jc, k, n, v_eff - take);
            }
          }
          __syncthreads();
#pragma unroll 1
          for (int jc = tid; jc < JA; jc += blockDim.x)
            if (s_mod[jc] && !(s_info[jc] & INFO_WIDE)) finish_row(jc);
          __syncthreads();
#pragma unroll 1
          for (int jc = warp; jc < JA; jc += nwarps)
            if (s_mod[jc] && (s_info[jc] & INFO_WIDE)) finish_wide(jc);
          __syncthreads();
        }
      }
      __syncthreads();

      // ---- fitness (Eq. 14) from the rows' terms, in the order of the dense kernel: per chunk of rows, thread
      // t adds rows t, t + 256, ... in double, a shuffle tree per warp, the warps in index order; then the
      // chunks in index order.  Published once all of the candidate's rows are written. ------------------
      if (tid < T) {
#pragma unroll 1
        for (int ch = 0; ch < a.chunks; ++ch) {
          const int j0 = ch * a.rows_per_chunk, j1 = min(J, j0 + a.rows_per_chunk);
          double acc = 0.0;
#pragma unroll 1
          for (int j = j0 + tid; j < j1; j += MAX_ROW_THREADS) acc += (double)s_term[j];
#pragma unroll
          for (int off = 16; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
          if (lane == 0) s_sums[ch * 8 + warp] = acc;
        }
      } else if (warp == T / 32) {
        // everybody's rows are written: made visible to the other blocks while the sums are formed
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
      }
#pragma unroll 1
      for (int i = tid; i < NN; i += blockDim.x) { s_tot[i] = 0; s_cnt[i] = 0u; s_viol[i] = 0; }
      if (tid == 0) { s_nmut2[set] = 0; s_nwide = 0; s_nslow = 0; s_nmod = 0; s_walk = 0; }
      __syncthreads();
      if (tid == T) {
        double sum = 0.0;
#pragma unroll 1
        for (int ch = 0; ch < a.chunks; ++ch) {
          double v[8], t = 0.0;
#pragma unroll
          for (int x = 0; x < 8; ++x) v[x] = s_sums[ch * 8 + x];
#pragma unroll
          for (int x = 0; x < 8; ++x) t += v[x];            // (warps that do not exist left zeros)
          sum += t;
        }
        const float f = fitness_finalise(a.tp.mode, a.tp.p, sum, (double)JA);
        const unsigned long long word = ((unsigned long long)(base + (uint32_t)s) << 32) | order_key(__float_as_uint(f));
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(pub_of(s, c)), "l"(word) : "memory");   // (behind this thread's fence)
        if (s == a.generations) a.fitness[c] = f;
      }
      ++item;
    }
}

// The best candidate (largest key, lowest index on ties) and its rows as a dense matrix; the next
// round's tags begin behind this round's.
__global__ void __launch_bounds__(256) flow_finish_kernel(FlowArgs a) {
  __shared__ unsigned long long s_best[8];
  __shared__ uint16_t s_place[FLOW_MAX_JOBS];      // place of a job's row, 0xFFFF: the job is not active
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, P = a.P, J = a.J, NN = a.NN, NS = wide_stride(NN);
  unsigned long long best = 0ull;
#pragma unroll 1
  for (int i = tid; i < P; i += 256) {
    const unsigned long long v = ((unsigned long long)order_key(__float_as_uint(a.fitness[i])) << 32) | (0xFFFFFFFFu - (uint32_t)i);
    best = v > best ? v : best;
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, off);
    best = o > best ? o : best;
  }
  if (lane == 0) s_best[warp] = best;
#pragma unroll 1
  for (int j = tid; j < J; j += 256) s_place[j] = 0xFFFFu;
  __syncthreads();
#pragma unroll 1
  for (int w = 0; w < 8; ++w) best = s_best[w] > best ? s_best[w] : best;
  const int found = (int)(0xFFFFFFFFu - (uint32_t)best), JA = *a.r.num_act;
  const int c = sched_index_ok(a.status, found >= 0 && found < P, SCHED_CHK_SLOT) ? found : 0;
#pragma unroll 1
  for (int i = tid; i < JA; i += 256) s_place[a.r.act[i]] = (uint16_t)i;
  __syncthreads();
  if (blockIdx.x == 0 && tid == 0) {
    *a.best_fitness = a.fitness[c];
    *a.r.base += (uint32_t)a.generations + 1u;
  }
  const size_t cand = (size_t)(a.generations & (DEPTH - 1)) * P + c;
#pragma unroll 1
  for (int j = blockIdx.x * 8 + warp; j < J; j += gridDim.x * 8) {
    const int jc = s_place[j];
    int16_t *out = a.best + (size_t)j * NN;
    Record r = {{NO_NODE, NO_NODE, NO_NODE, NO_NODE, NO_NODE, NO_NODE, 0u, 0u}};
    if (jc != 0xFFFF) r = load_record(a.r.rec + (cand * J + jc) * REC_WORDS);
    const int16_t *wide = a.r.wide + (cand * J + jc) * NS;
#pragma unroll 1
    for (int n = lane; n < NN; n += 32) {
      int v = 0;
      if (r.w[0] == WIDE) {
        v = wide[n];
      } else {
#pragma unroll
        for (int k = 0; k < ENTRIES; ++k) v = entry_node(r.w[k]) == n ? entry_gpus(r.w[k]) : v;
      }
      out[n] = (int16_t)v;
    }
  }
}

// the last population as dense matrices
__global__ void __launch_bounds__(256) flow_gather_kernel(FlowRows f, int P, int J, int NN, int generations, int16_t *__restrict__ out) {
  __shared__ uint16_t s_place[FLOW_MAX_JOBS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NS = wide_stride(NN), JA = *f.num_act;
#pragma unroll 1
  for (int j = tid; j < J; j += 256) s_place[j] = 0xFFFFu;
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < JA; i += 256) s_place[f.act[i]] = (uint16_t)i;
  __syncthreads();
  const size_t first = (size_t)(generations & (DEPTH - 1)) * P;
#pragma unroll 1
  for (long long row = (long long)blockIdx.x * 8 + warp; row < (long long)P * J; row += (long long)gridDim.x * 8) {
    const long long c = row / J;
    const int jc = s_place[row - c * J];
    Record r = {{NO_NODE, NO_NODE, NO_NODE, NO_NODE, NO_NODE, NO_NODE, 0u, 0u}};
    const size_t at = (first + c) * J + jc;
    if (jc != 0xFFFF) r = load_record(f.rec + at * REC_WORDS);
#pragma unroll 1
    for (int n = lane; n < NN; n += 32) {
      int v = 0;
      if (r.w[0] == WIDE) {
        v = f.wide[at * NS + n];
      } else {
#pragma unroll
        for (int k = 0; k < ENTRIES; ++k) v = entry_node(r.w[k]) == n ? entry_gpus(r.w[k]) : v;
      }
      out[row * NN + n] = (int16_t)v;
    }
  }
}

int flow_row_threads(int J) { return std::min(MAX_ROW_THREADS, (J + 31) & ~31); }
// row threads, the warp of the perturbed rows, and (ahead) as many threads again that draw the next step
int flow_threads(int J, bool ahead) { return flow_row_threads(J) * (ahead ? 2 : 1) + 32; }

}  // namespace

namespace {

// The pieces of the round's one allocation (tables and fitness among them); total with base NULL.
struct FlowArena {
  FlowRows r;
  float *goodput, *speedup, *speedup_rack, *fitness;
  size_t total;
};

FlowArena flow_arena(const sched_ctx *ctx, char *base) {
  const sched_config &c = ctx->cfg;
  const size_t P = c.population, J = c.num_jobs, NS = wide_stride(c.num_nodes), tab = J * ctx->KD * ctx->ND * 4;
  FlowArena f = {};
  size_t off = 0;
#define TAKE(field, type, bytes) do { f.field = (type *)(base + off); off += ((size_t)(bytes) + 255) & ~(size_t)255; } while (0)
  TAKE(goodput, float, tab);
  TAKE(speedup, float, tab);
  if (ctx->d_rack) TAKE(speedup_rack, float, tab);
  TAKE(fitness, float, P * 4);
  TAKE(r.cur_rec, uint32_t, 2 * J * REC_WORDS * 4);
  TAKE(r.same, uint32_t, J * REC_WORDS * 4);
  TAKE(r.pen, float, J * 4);
  TAKE(r.act, uint16_t, J * 2);
  TAKE(r.num_act, int, 4);
  TAKE(r.base, uint32_t, 4);
  TAKE(r.pub, unsigned long long, DEPTH * P * 8);
  TAKE(r.cur_wide, int16_t, 2 * J * NS * 2);
  TAKE(r.rec, uint32_t, DEPTH * P * J * REC_WORDS * 4);
  TAKE(r.wide, int16_t, DEPTH * P * J * NS * 2);
#undef TAKE
  f.total = off;
  return f;
}

constexpr int FLOW_OCC = 16;      // occupants listed per node: a group of lanes

size_t flow_smem_bytes(const sched_ctx *ctx, bool ahead) {
  int rows, chunks;
  fitness_chunking(ctx, ctx->cfg.population, rows, chunks);
  return flow_smem(ctx->cfg.population, ctx->cfg.num_jobs, ctx->cfg.num_nodes, FLOW_OCC,
                   flow_threads(ctx->cfg.num_jobs, ahead) / 32, chunks).total;
}

}  // namespace

// Blocks for this context's rounds (0: they run on the other kernels), and their allocation.  The rows
// of four generations with room for every row's contents may take half of the store's budget (a
// tighter budget is what the row pool is for), and all blocks must fit the GPU at once.
int round_flow_ensure(sched_ctx *ctx) {
  const sched_config &c = ctx->cfg;
  if (c.num_jobs < 1 || c.num_jobs > FLOW_MAX_JOBS || c.num_nodes > FLOW_MAX_NODES || ctx->cap_max > 2047) return SCHED_OK;
  const unsigned long long rows = (unsigned long long)DEPTH * c.population * c.num_jobs * (REC_WORDS * 4 + wide_stride(c.num_nodes) * 2);
  if (2 * rows > ctx->rs_budget) return SCHED_OK;
  int coop = 0, blocks = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess || !coop ||
      cudaFuncSetAttribute(flow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess) {
    cudaGetLastError();
    return SCHED_OK;
  }
  // threads that draw ahead where every candidate still has a block of its own (and its nodes' draws pay)
  for (int ahead = c.num_jobs <= SMEM_RECORDS ? 1 : 0; ahead >= 0; --ahead) {
    const size_t smem = flow_smem_bytes(ctx, ahead != 0);
    int per_sm = 0;
    if (smem > 220 * 1024 ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, flow_kernel, flow_threads(c.num_jobs, ahead != 0), smem) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    blocks = std::min(c.population, per_sm * ctx->num_sms);
    ctx->fl_ahead = ahead != 0;
    if (blocks == c.population) break;
  }
  if (blocks < 1) return SCHED_OK;
  const FlowArena size = flow_arena(ctx, nullptr);
  if (cudaMalloc((void **)&ctx->fl_arena, size.total) != cudaSuccess) {
    cudaGetLastError();
    ctx->fl_arena = nullptr;
    return SCHED_OK;
  }
  const FlowArena f = flow_arena(ctx, (char *)ctx->fl_arena);
  ctx->d_tab_goodput = f.goodput;
  ctx->d_tab_speedup = f.speedup;
  ctx->d_tab_speedup_rack = f.speedup_rack;
  ctx->d_fit_buf = ctx->d_fit = f.fitness;
  ctx->scratch_epoch++;
  // no tag matches before it is published, and a record that was never written has no nodes
  SCHED_CUDA_CHECK(ctx, cudaMemsetAsync(f.r.pub, 0, DEPTH * (size_t)c.population * 8, ctx->stream));
  SCHED_CUDA_CHECK(ctx, cudaMemsetAsync(f.r.base, 1, 4, ctx->stream));
  ctx->fl_blocks = blocks;
  return SCHED_OK;
}

static FlowArgs flow_args(const sched_ctx *ctx, const sched_jobs *jobs, const int16_t *d_cur) {
  const sched_config &c = ctx->cfg;
  FlowArgs a = {};
  a.r = flow_arena(ctx, (char *)ctx->fl_arena).r;
  a.cap = ctx->d_cap; a.k_cap = jobs->k_cap; a.active = jobs->active; a.cur = d_cur;
  a.age = jobs->age_sec; a.restarts = jobs->num_restarts; a.delta = c.delta_sec;
  a.rack = ctx->d_rack; a.table_rack = ctx->d_tab_speedup_rack;
  a.tp.table = ctx->d_tab_speedup;
  a.tp.pen = d_cur && jobs->age_sec && jobs->num_restarts ? a.r.pen : nullptr;
  a.tp.active = nullptr; a.tp.k_max = c.k_max; a.tp.n_max = c.n_max; a.tp.mode = fitness_mode(c.p); a.tp.p = c.p;
  a.tp.floor_ = c.speedup_floor;
  a.P = c.population; a.J = c.num_jobs; a.NN = c.num_nodes; a.k_max = c.k_max; a.n_max = c.n_max;
  a.num_elite = c.num_elite; a.occ = FLOW_OCC; a.row_threads = flow_row_threads(c.num_jobs);
  a.thr_init = c.thr_init; a.thr_mutate = c.thr_mutate;
  a.key = make_key(c.seed, ctx->d_round);
  fitness_chunking(ctx, c.population, a.rows_per_chunk, a.chunks);
  a.fitness = ctx->d_fit;
  a.wait_limit = ctx->fl_wait_limit;
  a.status = ctx->d_status;
  return a;
}

// The search of a round, after its tables.
int launch_round_flow(sched_ctx *ctx, const sched_jobs *jobs, const int16_t *d_cur, int32_t generations, int16_t *d_best,
                      float *d_best_fitness) {
  const sched_config &c = ctx->cfg;
  FlowArgs a = flow_args(ctx, jobs, d_cur);
  a.generations = generations;
  a.best = d_best; a.best_fitness = d_best_fitness;
  {
    TimedLaunch tl_(ctx, KK_FLOW_BUILD);
    flow_build_kernel<<<(c.num_jobs + 3) / 4, 128, 0, ctx->stream>>>(a);
  }
  SCHED_LAUNCH_CHECK(ctx);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)ctx->fl_blocks);
  lc.blockDim = dim3((unsigned)flow_threads(c.num_jobs, ctx->fl_ahead));
  lc.dynamicSmemBytes = flow_smem_bytes(ctx, ctx->fl_ahead);
  lc.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  {
    TimedLaunch tl_(ctx, KK_FLOW);
    SCHED_CUDA_CHECK(ctx, cudaLaunchKernelEx(&lc, flow_kernel, a));
  }
  SCHED_LAUNCH_CHECK(ctx);
  {
    TimedLaunch tl_(ctx, KK_FLOW_FINISH);
    flow_finish_kernel<<<std::min((c.num_jobs + 7) / 8, ctx->num_sms), 256, 0, ctx->stream>>>(a);
  }
  SCHED_LAUNCH_CHECK(ctx);
  ctx->fl_generations = generations;
  ctx->d_pop_last = (int16_t *)a.r.rec;
  return SCHED_OK;
}

int flow_gather(sched_ctx *ctx, int16_t *d_out) {
  const sched_config &c = ctx->cfg;
  const long long want = ((long long)c.population * c.num_jobs + 7) / 8;
  {
    TimedLaunch tl_(ctx, KK_FLOW_GATHER);
    flow_gather_kernel<<<(unsigned)std::min<long long>(want, (long long)ctx->num_sms * 8), 256, 0, ctx->stream>>>(
        flow_arena(ctx, (char *)ctx->fl_arena).r, c.population, c.num_jobs, c.num_nodes, ctx->fl_generations, d_out);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}
