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
// Rows of inactive jobs are left out.  One block works on one candidate at a time: a thread per row that is copied as it
// is; eight lanes per row that is perturbed or that the repair changes, an entry each, so that what is done
// to a row's nodes is done to all of them at once, four rows a warp (a thread per row where there are very many).  Warps of their own draw a step ahead.
// Bound: the length of a block's chain of steps.  A generation of the testbed (48 jobs x 100 candidates) in cycles,
// 7.2 k in all: waiting for the four keys 1.4 k (an unloaded L2 trip is 0.3 k; a fence behind a store 0.8 k), parents
// 0.35 k, perturbed rows 1.9 k, decisions 1.4 k, changed rows 0.85 k, sum and power mean 1.15 k beside the fence
// (0.95 k), publication 0.2 k.  13 k before perturbed and changed rows took eight lanes, draws and terms moved out of
// the way and keys apart.  Eight lanes for the rows that are copied, too: 1.08 times the time of the testbed's round and twice
// that of the large one (both measured before the keys were set apart), four times the instructions for as many rows.
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
// Words from one candidate's published key to the next's.  Side by side, a hundred keys are seven lines that
// every block polls, and polls and publications queue there: testbed round 494 us, 422 with 32 bytes between them, 415 with
// 64, 420 with 128; 210 jobs x 150 candidates 708, 555, 549, 565; racks 528, 449, 438, 438.
constexpr int PUB_STRIDE = 8;
constexpr int SUM_THREADS = 256;                // as the dense fitness kernel: the order of its sums
constexpr int LANES = 8;                        // lanes of a row
constexpr int STASH = 256;                      // perturbed rows of many whose draws are kept, further ones draw again
constexpr int SMEM_RECORDS = 256;              // up to this many jobs the child's records are kept in shared memory, too
constexpr int FLOW_MAX_WARPS = 20;
// With more generations than this, or with so few jobs and no fewer generations than jobs, a block copies the rows' terms to
// shared memory where they fit.  The copy takes 0.11 us a job, a generation then up to 0.27 us less: 8 candidates x 200 jobs, none, 10 and
// 100 generations with the copy 54, 96 and 466 us, without 32, 79 and 470; 148 x 250 63, 113 and 543, 36, 89 and 542; 100 x 48
// 34, 73 and 419, 30, 67 and 414; but 59 x 18, 30 generations, 122 and 126, 32 x 8, 10 generations, 55.1 and 55.8.
constexpr int TERMS_FROM = 100, TERMS_JOBS = 40;
// More perturbed or changed rows a warp than this have a thread each instead of eight lanes, in blocks of many jobs that share their SM:
// three rounds of four rows take a warp longer than one of 32, and the issue slots are full.  30 generations of 512 candidates x
// 1024 jobs on 64 nodes, a tenth of the rows perturbed 1329 us with eight lanes, 1124, a fifth 1795, 1332; 832 x 2224, a fifth 6035, 4257.
constexpr int LISTS_FROM = 12;
constexpr int MANY_TWO_JOBS = 2048;             // beyond these two blocks an SM take any population
constexpr int SOME_WARPS = 16;                  // that work on the rows where a block has an SM for itself and more than 256 jobs
constexpr int FLOW_OCC = 16;                    // occupants of a node that a group of lanes decides
constexpr int FLOW_MAX_JOBS = 8192, FLOW_MAX_NODES = 512, FLOW_MAX_SMEM = 220 * 1024;
constexpr int RANK_PAIRS = 64;                 // keys that are ranked by comparing them with one another

// Kinds of the generation kernel.  Not MANY, MANY_TWO: the child's records and what its rows' terms are made of are kept in
// shared memory, too.  FEW_ALONE, SOME_ALONE: no two blocks share an SM (a population of at most as many), up to 256 jobs and
// up to what the memory holds (some 2700).  FEW: two blocks, or more with up to 256 jobs.  MANY_TWO: two blocks, or one with more
// jobs than SOME_ALONE holds, and any number of candidates beyond 2048 jobs, where four blocks an SM have more records between
// them than L2 holds and take more turns than their number saves (592 candidates x 2500 jobs 2441 us with MANY, 2312; 900 x 3000
// 7247, 5472; 592 x 1500 2483, 2663).  Registers: 138 for FEW_ALONE's 12 warps (with 96 a testbed round takes 1.07 times as long, with 64
// 1.13 times: spills lie in the L1 that every acquire empties; measured before the keys were set apart), 96 for SOME_ALONE's 20, 64
// for FEW and MANY_TWO, 56 for MANY.  A lone candidate's block with more than 1024 jobs had 8 or 9 warps, which is 30 generations
// of 64 x 1100 jobs 1028 us, now 642; 148 x 4000 2206, now 1374; 296 x 2400 1854, now 1135.
// CROWDED, with any of them: lists longer than a group of lanes, where so many occupants of a node are to be expected.
constexpr int FEW_ALONE = 0, SOME_ALONE = 1, FEW = 2, MANY = 3, MANY_TWO = 4, CROWDED = 8;
__host__ __device__ constexpr int shape_of(int kind) { return kind & 7; }
__host__ __device__ constexpr bool few(int kind) { return shape_of(kind) < MANY; }
__host__ __device__ constexpr int kind_threads(int kind) {
  return shape_of(kind) == FEW_ALONE ? 384 : shape_of(kind) == SOME_ALONE ? 640 : shape_of(kind) == MANY ? 288 : 512;
}
__host__ __device__ constexpr int kind_blocks(int kind) { return shape_of(kind) == MANY ? 4 : shape_of(kind) <= SOME_ALONE ? 1 : 2; }

__host__ __device__ inline int wide_stride(int NN) { return (NN + 7) & ~7; }
__host__ __device__ inline int stash_rows(int J) { return J <= SMEM_RECORDS ? J : STASH; }

struct FlowRows {
  uint32_t *rec;             // [DEPTH][P][J][REC_WORDS]; rows of active jobs only, one behind the other
  int16_t *wide;             // [DEPTH][P][J][wide_stride] contents of wide rows
  uint32_t *cur_rec;         // [2][J][REC_WORDS] the current allocation after the row caps, and before them
  int16_t *cur_wide;         // [2][J][wide_stride]
  uint32_t *same;            // [J][REC_WORDS] a row that counts as unchanged, with its term (first entry NEVER: there is none
                             // with six nodes or fewer)
  float *terms;              // [J][classes][k_max + 1] term of a row that counts as changed (or of any, without the penalty), by
                             // its GPUs and where they are: one node, several, several racks
  float *pen;                // [J] penalty factor of a row that differs from the current allocation's
  uint16_t *act;             // [J] active jobs, ascending; act[J] .. : see num_act
  int *num_act;
  unsigned long long *pub;   // [DEPTH][P][PUB_STRIDE] tag << 32 | fitness key
  uint32_t *base;            // tag of the round's initial population
};
constexpr uint32_t NEVER = 0xFFFFFFFDu;

// Places in the generation kernel's shared memory, behind what the warps tell each other (terms: -1 where they are not kept there).
struct FlowSmem {
  int act, term, info, node, occ, more, viol, cap, rack, mut, mod, stash, flag, dense, rep, keys, sums, scratch, rec, same,
      terms, total;
};

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
  const int32_t *nmin;       // [k_max + 1] fewest nodes, two or more, that K replicas fit on
  int P, J, NN, k_max, n_max, num_elite, generations;
  int warps;                 // warps that work on the rows; the others draw
  int more;                  // occupants listed per node beyond FLOW_OCC
  int classes;               // 2, or 3 with racks
  FlowSmem at;
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
// The word (tag << 32 | key) published under `tag`; 0 when it has not come within the limit (the caller returns: the
// other blocks' waits run out the same way).  A thread that has waited calls waited() before the barrier
// behind which the block reads the rows, or before it publishes in its turn.
__device__ __forceinline__ unsigned long long wait_tag(const unsigned long long *p, uint32_t tag, unsigned int limit, int *status) {
#pragma unroll 1
  for (unsigned int n = 0; n < limit; ++n) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    if ((uint32_t)(v >> 32) == tag) return v;
  }
  atomicCAS(status, 0, SCHED_ERR_TIMEOUT);
  return 0ull;
}
// Acquire: with the publisher's fence (release) and the block's barrier, what was written before the tag
// was published is seen by every thread of this block, and what was read before it lies behind it.  One
// fence after the polls that succeeded, not an acquire in each poll.  The one-way fence costs nothing that
// can be measured, fence.acq_rel, which also waits for this thread's own writes, 10 % of a testbed round and 4 % of a
// large one (of rounds that took 663 us and 3.87 ms).
__device__ __forceinline__ void waited() { asm volatile("fence.acquire.gpu;" ::: "memory"); }
__device__ __forceinline__ void publish(unsigned long long *p, uint32_t tag, uint32_t key) {
  const unsigned long long v = ((unsigned long long)tag << 32) | key;
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// ---- fitness terms of rows laid out in shared memory ----------------------------------------------
// table of a row by the racks its nodes lie in
__device__ __forceinline__ const float *table_of(const FlowArgs &a, int lo, int hi) { return lo < hi ? a.table_rack : a.tp.table; }

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
#pragma unroll 1
    for (unsigned left = m; left && base < ENTRIES; left &= left - 1u, ++base) {
      const int at = __ffs(left) - 1;
      const uint32_t e = ((uint32_t)(n0 + at) << 16) | (uint32_t)__shfl_sync(0xffffffffu, v, at);
      if (lane == base) mine = e;
    }
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
  // (not through the read-only path: flow_build_kernel calls this, and the tables' kernel writes them while it runs)
  const float sp = __ldcg(table_of(a, lo, hi) + fitness_table_index(a.tp, j, K, N));
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
#pragma unroll 8
    for (int j0 = 0; j0 < J; j0 += 32) {
      const bool on = j0 + lane < J && (!a.active || __ldg(a.active + j0 + lane));
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
    const float pen = a.tp.pen && raw > 0 ? realloc_factor(a.age[j], a.restarts[j], a.delta) : 1.f;
    if (a.tp.pen && lane == 0) a.r.pen[j] = pen;
    __syncwarp();
    int K, N;
    dense_totals(row, NN, lane, K, N);
    asm volatile("griddepcontrol.wait;" ::: "memory");      // the tables
    // (what a row of the search can be: on one node, or on as many as its GPUs need at least; the table has one
    // value for all of those)
    const int KD = a.k_max + 1, ND = a.n_max + 1;
#pragma unroll 2
    for (int k = lane; k < KD; k += 32) {
      const int many = k >= 2 ? __ldg(a.nmin + k) : ND, one = k >= 1 ? 1 : ND;
      const size_t from = ((size_t)j * KD + k) * ND;
      float *to = a.r.terms + (size_t)j * a.classes * KD + k;
      const float x0 = one < ND ? __ldcg(a.tp.table + from + one) : 0.f, x1 = many < ND ? __ldcg(a.tp.table + from + many) : 0.f;
      const float x2 = a.classes > 2 && many < ND ? __ldcg(a.table_rack + from + many) : 0.f;
      to[0] = fitness_term_with(a.tp, x0, pen, true);
      to[KD] = fitness_term_with(a.tp, x1, pen, true);
      if (a.classes > 2) to[2 * KD] = fitness_term_with(a.tp, x2, pen, true);
    }
    const int kc = max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max));
    Record r;
#pragma unroll 1
    for (int caps = 1; caps >= 0; --caps) {     // before the caps (the second set), then after them (the first)
      const bool over = K > kc || N > a.n_max;
      if (!caps) dense_caps(row, NN, K, N, kc, a.n_max, lane);
      const size_t at = (size_t)caps * J + j;
      if (caps || over || N > ENTRIES) r = dense_record(a, row, j, K, N, a.r.cur_wide + at * NS, lane);
      if (lane == 0) store_record(a.r.cur_rec + at * REC_WORDS, r);
      if (caps && lane == 0) {
        Record same = r;
        if (!a.tp.pen || !in_range || N > ENTRIES) same.w[0] = NEVER;
        store_record(a.r.same + (size_t)j * REC_WORDS, same);
      }
      __syncwarp();
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");        // (a block without an active job ends after the tables, too)
}

constexpr int INFO_DIST = 1;        // the row spanned two nodes or more after the row pass (interference snapshot)
constexpr int INFO_CHANGED = 2;     // a node's decision changes it
constexpr int INFO_WIDE = 4;
constexpr int INFO_AGAIN = 8;       // a crowded node's decision changes it

// The candidate a block is working on.
struct Work {
  int src[2];                         // parents' first rows, counted in records from the population's first (initial population:
                                      // the current allocation's rows after and before the caps, by job)
  int dst;                            // the child's first row
  uint32_t c, gen;
  bool init;
};

// What the warps of a block tell each other.  Two sets where a candidate's draws are made while the one before
// it is worked on.
struct FlowCtl {
  int4 hand[2];                       // parents' first rows, 0: a wait ran out
  int nmut[2];
  int nwide, nslow, nmod, walk, po;
  uint32_t sel[2][4];
  unsigned long long word;            // what is published
  int red[FLOW_MAX_WARPS];
};

// The block's shared memory.
struct FlowView {
  FlowCtl &ctl;
  uint16_t *act;                      // active jobs
  float *term;                        // by job, 0 where there is none
  uint8_t *info;                      // by row
  uint32_t *node;                     // by node: GPUs placed on it; distributed jobs on it | occupants << 16
  uint32_t *occ;                      // row | GPUs << 13 | place in the record (7: wide) << 25 | distributed << 31
  uint32_t *more;                     // those that do not fit
  uint8_t *viol;                      // the node's column is to be walked
  int16_t *cap, *rack;
  uint16_t *mut;                      // two sets
  uint16_t *mod;                      // rows that decisions change
  uint16_t *wide;                     // in the same place, before the decisions: wide rows from the front, slow ones from the back
  uint2 *stash;                       // two sets: the draw that chooses a node of the row; operator | node << 2 | replica cap << 16
  uint8_t *flag;                      // two sets, by row: 1 from the second parent, 2 perturbed
  int16_t *dense;                     // a row per warp
  uint32_t *rep;                      // two sets, by node: the two rotation offsets
  uint32_t *keys;
  double *sums;
  uint32_t *scratch;                  // a record's place per eight lanes
  uint32_t *rec, *same;               // by row: the child's records, the unchanged rows (few jobs)
  float *terms;                       // by row (where they fit)
};

// (memory: its address in the shared window, so that functions that are called know what it points to)
__device__ __forceinline__ FlowView flow_view(const FlowArgs &a, uint32_t memory) {
  const FlowSmem &L = a.at;
  unsigned char *const s = (unsigned char *)__cvta_shared_to_generic(memory);
  return FlowView{*(FlowCtl *)s, (uint16_t *)(s + L.act), (float *)(s + L.term), s + L.info, (uint32_t *)(s + L.node),
                  (uint32_t *)(s + L.occ), (uint32_t *)(s + L.more), s + L.viol, (int16_t *)(s + L.cap), (int16_t *)(s + L.rack),
                  (uint16_t *)(s + L.mut), (uint16_t *)(s + L.mod), (uint16_t *)(s + L.mod),
                  (uint2 *)(s + L.stash), s + L.flag, (int16_t *)(s + L.dense), (uint32_t *)(s + L.rep), (uint32_t *)(s + L.keys),
                  (double *)(s + L.sums), (uint32_t *)(s + L.scratch), (uint32_t *)(s + L.rec), (uint32_t *)(s + L.same),
                  (float *)(s + L.terms)};
}

__device__ __forceinline__ uint32_t *rec_row(const FlowArgs &a, int row) { return a.r.rec + (ptrdiff_t)row * REC_WORDS; }
__device__ __forceinline__ int16_t *wide_row(const FlowArgs &a, int row) { return a.r.wide + (ptrdiff_t)row * wide_stride(a.NN); }
// contents of row jc (job j) of a parent
__device__ __forceinline__ const int16_t *wide_source(const FlowArgs &a, const Work &w, int from, int jc, int j) {
  return w.init ? a.r.cur_wide + ((size_t)from * a.J + j) * wide_stride(a.NN) : wide_row(a, (from ? w.src[1] : w.src[0]) + jc);
}

// The candidate of rank c (fitness key descending, index ascending) of P keys in shared memory, by one warp.
//
// By bits: the key, no less than `low` and no more than `high`, a bit and a pass over the keys at a time, then the
// one wanted of those that have it.
__device__ __noinline__ int candidate_by_bits(const uint32_t *key, int P, int c, uint32_t low, uint32_t high, int lane) {
  const int bits = 32 - __clz((int)(low ^ high));         // (what the two have in common the key has, too)
  uint32_t found = bits < 32 ? high >> bits << bits : 0u;
#pragma unroll 1
  for (uint32_t bit = bits ? 1u << (bits - 1) : 0u; bit; bit >>= 1) {
    const uint32_t want = (found | bit), mask = 0u - bit;      // the bits known so far, and this one set
    int n = 0;
#pragma unroll 4
    for (int i = lane; i < P; i += 32) n += (key[i] & mask) == want ? 1 : 0;
    n = __reduce_add_sync(0xffffffffu, n);
    if (c < n) found = want;
    else c -= n;
  }
  int at = 0x7fffffff;
#pragma unroll 1
  for (int i0 = 0; i0 < P; i0 += 32) {
    const bool equal = i0 + lane < P && key[i0 + lane] == found;
    const unsigned m = __ballot_sync(0xffffffffu, equal);
    if (equal && __popc(m & ((1u << lane) - 1u)) == c) at = i0 + lane;
    c -= __popc(m);
    if (c < 0) break;
  }
  return __reduce_min_sync(0xffffffffu, at);
}
// The (c + 1)-th largest of the lanes' own maxima is no larger than the key wanted, so only the keys from there
// on (about twice c) are ranked, by comparing them with one another; list: room for P.  That is quicker for up
// to 64 of them (31 elite candidates of 100: 608 us a round of the testbed, by bits 875), and takes the square of their
// number: where it took all of them, which ranks from the 33rd on and populations that have converged to a few
// fitness values did, the round took 21.8 ms for 512 candidates of the testbed (now 1.23 ms with 40 elite ones,
// 0.63 ms if all are equal) and 340 ms for 2048 (4.2 and 2.0 ms).  100 candidates, all equal: by pairs 1440 us, 420 by bits.
__device__ __noinline__ int candidate_of_rank(const uint32_t *key, int P, int c, uint16_t *list, int lane) {
  if (c >= 32) return candidate_by_bits(key, P, c, 0u, 0xFFFFFFFFu, lane);
  uint32_t top = 0u;
#pragma unroll 4
  for (int i = lane; i < P; i += 32) top = max(top, key[i]);
  int before = 0;                       // lanes whose maximum comes first
#pragma unroll 1
  for (int l = 0; l < 32; ++l) {
    const uint32_t o = __shfl_sync(0xffffffffu, top, l);
    before += o > top || (o == top && l < lane) ? 1 : 0;
  }
  const uint32_t bound = __shfl_sync(0xffffffffu, top, __ffs(__ballot_sync(0xffffffffu, before == c)) - 1);
  int n = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < P; i0 += 32) {
    const bool in = i0 + lane < P && key[i0 + lane] >= bound;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (in) list[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(i0 + lane);
    n += __popc(m);
  }
  if (n > RANK_PAIRS) return candidate_by_bits(key, P, c, bound, __reduce_max_sync(0xffffffffu, top), lane);
  __syncwarp();
  int found = 0x7fffffff;
#pragma unroll 1
  for (int x = lane; x < n; x += 32) {
    const int i = list[x];
    const uint32_t k = key[i];
    int rank = 0;
#pragma unroll 2
    for (int y = 0; y < n; ++y) {
      const uint32_t o = key[list[y]];
      rank += o > k || (o == k && y < x) ? 1 : 0;
    }
    if (rank == c) found = i;
  }
  return __reduce_min_sync(0xffffffffu, found);
}

// Barriers: 0 is the whole block's.
constexpr int BAR_ROWS = 1;           // the warps that work on rows
constexpr int BAR_SUMS = 2;           // all of them but the last
constexpr int BAR_KEY = 3;            // the first and the last of them
__device__ __forceinline__ void bar(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

// Minimum and exclusive prefix sum over the warps that work on rows; both end with a barrier.
__device__ __noinline__ int block_min(int v, int *s_red, int nwarps) {
  v = __reduce_min_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  bar(BAR_ROWS, nwarps * 32);
  int r = s_red[0];
#pragma unroll 1
  for (int w = 1; w < nwarps; ++w) r = min(r, s_red[w]);
  bar(BAR_ROWS, nwarps * 32);
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
  bar(BAR_ROWS, nwarps * 32);
  int before = 0;
  total = 0;
#pragma unroll 1
  for (int w = 0; w < nwarps; ++w) {
    const int t = s_red[w];
    if (w < warp) before += t;
    total += t;
  }
  bar(BAR_ROWS, nwarps * 32);
  return before + incl - v;
}

// GPUs of a finished row of this block's candidate on a node
template <int KIND>
__device__ __noinline__ int row_at(const FlowArgs &a, int row, int node) {
  const Record r = load_record(rec_row(a, row));
  if (r.w[0] == WIDE) return (int)__ldcg(wide_row(a, row) + node);
  int v = 0;
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k) v = entry_node(r.w[k]) == node ? entry_gpus(r.w[k]) : v;
  return v;
}

// ---- rows, eight lanes each: lane k has word k of the record --------------------------------------
// Called by whole warps; `live`: this lane's row is one.

// of a warp's ballot, the bits of this lane's row
__device__ __forceinline__ unsigned row_bits(bool p, int lane) { return (__ballot_sync(0xffffffffu, p) >> (lane & 24)) & 0xFFu; }

__device__ __forceinline__ int row_sum(int v) {
#pragma unroll
  for (int off = LANES / 2; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// a row's occupant into the nodes' totals and lists
template <int KIND>
__device__ __forceinline__ void add_occupant(const FlowArgs &a, const FlowView &v, int jc, int k_rec, uint32_t e, bool dist) {
  const int n = entry_node(e);
  if (!sched_index_ok(a.status, n < a.NN && jc < a.J && entry_gpus(e) <= 2047, SCHED_CHK_NODE)) return;
  atomicAdd(&v.node[2 * n], (uint32_t)entry_gpus(e));
  const uint32_t k = atomicAdd(&v.node[2 * n + 1], (dist ? 1u : 0u) | (1u << 16)) >> 16;
  auto entry = [&] { return (uint32_t)jc | ((uint32_t)entry_gpus(e) << 13) | ((uint32_t)k_rec << 25) | (dist ? 0x80000000u : 0u); };
  if (k < (uint32_t)FLOW_OCC) v.occ[n * FLOW_OCC + k] = entry();
  else if constexpr ((KIND & CROWDED) != 0)
    if (k < (uint32_t)(FLOW_OCC + a.more)) v.more[n * a.more + (int)k - FLOW_OCC] = entry();
}

// A word of a finished row goes to its place: the child's records, the term by job.
template <int KIND>
__device__ __forceinline__ void put_word(const FlowArgs &a, const FlowView &v, int dst, int jc, int k, uint32_t word) {
  rec_row(a, dst + jc)[k] = word;
  if (few(KIND)) v.rec[jc * REC_WORDS + k] = word;
  if (k == REC_TERM) v.term[v.act[jc]] = __uint_as_float(word);
}

// Eight words of a warp's own, for a row whose entries are to be put in order: emptied, filled (by all lanes of the row that
// have one), read.
__device__ __forceinline__ uint32_t *empty_place(const FlowView &v, int warp, int lane) {
  uint32_t *place = v.scratch + warp * 32 + (lane & 24);
  place[lane & 7] = NO_NODE;
  __syncwarp();
  return place;
}

// A row's finished list becomes its record, the term from the classes' terms or the unchanged row's; in the row pass
// (`fresh`) its occupants are added up.  e: this lane's entry, in any order; K, N: their GPUs and number; place: the entries in
// order.
template <int KIND>
__device__ __forceinline__ void settle_row(const FlowArgs &a, const FlowView &v, int dst, int jc, uint32_t e, const uint32_t *place, int K, int N,
                                           bool live, bool fresh, int lane) {
  const int k = lane & 7;
  int cls = N >= 2 ? 1 : 0;
  if (a.rack) {
    const bool on = e != NO_NODE && sched_index_ok(a.status, entry_node(e) < a.NN, SCHED_CHK_NODE);
    const int r = on ? (int)v.rack[entry_node(e)] : -1;
    const unsigned have = row_bits(on, lane);
    const int first = __shfl_sync(0xffffffffu, r, have ? __ffs(have) - 1 : 0, LANES);
    if (row_bits(on && r != first, lane)) cls = 2;
  }
  if (!live || !sched_index_ok(a.status, K >= 0 && K <= a.k_max && jc < a.J, SCHED_CHK_ENTRY)) K = 0;
  const int row = a.classes * (a.k_max + 1), at = cls * (a.k_max + 1) + K, j = v.act[jc];
  const uint32_t same = few(KIND) ? v.same[jc * REC_WORDS + k] : __ldg(a.r.same + (size_t)j * REC_WORDS + k);
  const float changed = few(KIND) && a.at.terms >= 0 ? v.terms[jc * row + at] : __ldg(a.r.terms + (size_t)j * row + at);
  __syncwarp();
  const uint32_t word = place[k];
  const uint32_t unchanged = __shfl_sync(0xffffffffu, same, REC_TERM, LANES);
  const bool equal = (row_bits(word == same, lane) & 0x3Fu) == 0x3Fu;
  if (live) {
    put_word<KIND>(a, v, dst, jc, k, k < ENTRIES ? word : k == REC_TERM ? (equal ? unchanged : __float_as_uint(changed)) : 0u);
    if (fresh && k < ENTRIES && word != NO_NODE) add_occupant<KIND>(a, v, jc, k, word, N >= 2);
    if (fresh && k == 0) v.info[jc] = N >= 2 ? INFO_DIST : 0;
  }
  __syncwarp();
}

// Row caps: replicas above kc leave from the highest node index down, then occupied nodes beyond n_max from the
// highest index down.  The list in place; its GPUs and entries then.
__device__ __noinline__ int2 cap_list(uint32_t *place, int K, int N, int kc, int n_max, bool over, int lane) {
  __syncwarp();
  const int k = lane & 7;
  uint32_t e = place[k];
  const int gpus = e != NO_NODE ? entry_gpus(e) : 0;
  int upto = gpus;
#pragma unroll
  for (int off = 1; off < LANES; off <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, upto, off, LANES);
    if (k >= off) upto += u;
  }
  if (over && e != NO_NODE) {
    const int take = min(gpus, max(upto - kc, 0));
    e = take == gpus || k >= n_max ? NO_NODE : e - (uint32_t)take;
    place[k] = e;
  }
  return make_int2(row_sum(e != NO_NODE ? entry_gpus(e) : 0), __popc(row_bits(e != NO_NODE, lane)));
}

// What a row's draw says that its parent's contents do not change: the operator, the node it goes to; and the row's cap.
__device__ __forceinline__ uint2 choices_of(const FlowArgs &a, const u32x4 &m, int j) {
  const int cap = max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max));
  return make_uint2(m.z, bounded(m.y, 3u) | (bounded(m.w, (uint32_t)a.NN) << 2) | ((uint32_t)cap << 16));
}
static_assert(FLOW_MAX_NODES <= 512 && SCHED_MAX_K < 65536, "the choices' fields");

// The row pass for up to four perturbed rows: perturbation (grow, shrink, relocate, chosen by the row's draw), row caps,
// the new record.  x0: the first of them in the list.
template <int KIND>
__device__ __forceinline__ void perturb_rows(const FlowArgs &a, const FlowView &v, const Work &w, uint32_t round, int set, int x0, int nmut,
                                             int warp, int lane) {
  uint32_t *const place = empty_place(v, warp, lane);
  const int k = lane & 7, i = x0 + (lane >> 3);
  const unsigned below = (1u << k) - 1u;
  bool live = i < nmut;
  const int m = live ? v.mut[set * a.J + i] : 0, jc = m & 0x7FFF;
  live = live && sched_index_ok(a.status, i < a.J && jc < a.J, SCHED_CHK_LIST);
  uint32_t e = NO_NODE;
  if (live && k < ENTRIES) e = __ldcg(rec_row(a, (w.init || (m >> 15) ? w.src[1] : w.src[0]) + (w.init ? (int)v.act[jc] : jc)) + k);
  uint2 st = make_uint2(0u, 0u);
  if (live && i < stash_rows(a.J)) {
    st = v.stash[set * stash_rows(a.J) + i];
  } else if (live) {
    const int j = v.act[jc];
    st = choices_of(a, draw_one(a.key.k0, round, (uint32_t)j, w.c, w.gen, w.init ? SLOT_INIT : SLOT_MUTATE), j);
  }
  __syncwarp();
  const uint32_t op = st.y & 3u;
  const int nd = (int)((st.y >> 2) & 0x1FFu), cap_nd = (int)v.cap[nd], k_cap = (int)(st.y >> 16);
  const bool wide = (row_bits(k == 0 && e == WIDE, lane) & 1u) != 0u;
  int N = __popc(row_bits(e != NO_NODE, lane));
  const uint32_t es = __shfl_sync(0xffffffffu, e, N > 0 ? (int)bounded(st.x, (uint32_t)N) : 0, LANES);
  const int ns = entry_node(es), vs = entry_gpus(es);
  const unsigned at_nd = row_bits(e != NO_NODE && entry_node(e) == nd, lane);
  const uint32_t end = __shfl_sync(0xffffffffu, e, at_nd ? __ffs(at_nd) - 1 : 0, LANES);
  const int v_nd = at_nd ? entry_gpus(end) : 0;
  const bool change = op == 0u || (N > 0 && (op == 1u || nd != ns));
  const int X = op == 1u ? ns : nd, V = op == 0u ? min(v_nd + 1, cap_nd) : op == 1u ? vs - 1 : min(v_nd + vs, cap_nd);
  const uint32_t x = ((uint32_t)X << 16) | (uint32_t)V;
  const bool insert = change && op != 1u && !at_nd && V > 0;
  if (change && e != NO_NODE) {
    if (entry_node(e) == X) e = V > 0 ? x : NO_NODE;
    else if (op == 2u && entry_node(e) == ns) e = NO_NODE;
  }
  const unsigned there = row_bits(e != NO_NODE, lane);
  const int extra = insert ? 1 : 0, extra_at = __popc(row_bits(e != NO_NODE && e < x, lane));
  if (e != NO_NODE) place[__popc(there & below) + (e > x ? extra : 0)] = e;
  if (insert && k == 7) {                     // (a record has no seventh entry: the lane of the new one)
    place[extra_at] = x;
    e = x;
  }
  int K = row_sum(e != NO_NODE ? entry_gpus(e) : 0);
  N = __popc(there) + extra;
  const bool over = live && !wide && (K > k_cap || N > a.n_max);
  if (__any_sync(0xffffffffu, over)) {
    const int2 now = cap_list(place, K, N, k_cap, a.n_max, over, lane);
    K = now.x;
    N = now.y;
    __syncwarp();
    e = place[k];
  }
  const bool slow = live && (wide || N > ENTRIES);
  live = live && !slow;
  if (slow && k == 0) {
    const int at = atomicAdd(&v.ctl.nslow, 1);
    if (sched_index_ok(a.status, at < a.J, SCHED_CHK_LIST)) v.wide[a.J - 1 - at] = (uint16_t)m;
  }
  settle_row<KIND>(a, v, w.dst, jc, live ? e : NO_NODE, place, K, N, live, true, lane);
}

// A row without the entries that decisions took out (0 GPUs), and its new term.
template <int KIND>
__device__ __forceinline__ void finish_row(const FlowArgs &a, const FlowView &v, int dst, int jc, bool live, int warp, int lane) {
  uint32_t *const place = empty_place(v, warp, lane);
  const int k = lane & 7;
  uint32_t e = NO_NODE;
  if (live && k < ENTRIES) e = few(KIND) ? v.rec[jc * REC_WORDS + k] : __ldcg(rec_row(a, dst + jc) + k);
  if (entry_gpus(e) == 0) e = NO_NODE;
  const unsigned there = row_bits(e != NO_NODE, lane);
  if (e != NO_NODE) place[__popc(there & ((1u << k) - 1u))] = e;
  settle_row<KIND>(a, v, dst, jc, e, place, row_sum(e != NO_NODE ? entry_gpus(e) : 0), __popc(there), live, false, lane);
}

// ---- rows, a thread each: a third of the instructions that eight lanes take for a row, and a longer chain ------------
// Where a block has many such rows for its warps and shares its SM's issue slots with others.
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

// `gpus` of a node: the entry replaced, put in its place or taken out
__device__ __forceinline__ void list_set(uint32_t (&e)[LIST], int node, int gpus) {
  bool found = false;
  const uint32_t entry = gpus > 0 ? ((uint32_t)node << 16) | (uint32_t)gpus : NO_NODE;
#pragma unroll
  for (int k = 0; k < LIST; ++k)
    if (entry_node(e[k]) == node) {
      found = true;
      e[k] = entry;
    }
  uint32_t x = found ? NO_NODE : entry;
#pragma unroll
  for (int k = 0; k < LIST; ++k) {      // a new entry to its place, then a hole to the end
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

// As settle_row, for a list of up to six entries in order.
template <int KIND>
__device__ __forceinline__ void settle_list(const FlowArgs &a, const FlowView &v, int dst, int jc, const uint32_t (&e)[LIST], int K, int N, bool fresh) {
  const int j = v.act[jc], row = a.classes * (a.k_max + 1);
  int cls = N >= 2 ? 1 : 0;
  if (a.rack) {
    int first = -1;
#pragma unroll
    for (int k = 0; k < ENTRIES; ++k)
      if (e[k] != NO_NODE && sched_index_ok(a.status, entry_node(e[k]) < a.NN, SCHED_CHK_NODE)) {
        const int r = (int)v.rack[entry_node(e[k])];
        if (first < 0) first = r;
        if (r != first) cls = 2;
      }
  }
  if (!sched_index_ok(a.status, K >= 0 && K <= a.k_max && jc < a.J, SCHED_CHK_ENTRY)) return;
  const uint4 lo = __ldg((const uint4 *)(a.r.same + (size_t)j * REC_WORDS)), hi = __ldg((const uint4 *)(a.r.same + (size_t)j * REC_WORDS) + 1);
  const float changed = __ldg(a.r.terms + (size_t)j * row + cls * (a.k_max + 1) + K);
  if (fresh) {
    v.info[jc] = N >= 2 ? INFO_DIST : 0;
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
      uint32_t x = e[0];
#pragma unroll
      for (int z = 1; z < ENTRIES; ++z) x = z == k ? e[z] : x;
      add_occupant<KIND>(a, v, jc, k, x, N >= 2);
    }
  }
  const bool equal = lo.x == e[0] && lo.y == e[1] && lo.z == e[2] && lo.w == e[3] && hi.x == e[4] && hi.y == e[5];
  Record r;
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k) r.w[k] = e[k];
  r.w[REC_TERM] = equal ? hi.z : __float_as_uint(changed);
  r.w[7] = 0u;
  store_record(rec_row(a, dst + jc), r);
  v.term[j] = __uint_as_float(r.w[REC_TERM]);
}

// As perturb_rows, for up to 32 rows.
template <int KIND>
__device__ __noinline__ void perturb_lists(const FlowArgs &a, uint32_t memory, Work w, uint32_t round, int set, int x0, int nmut, int lane) {
  const FlowView v = flow_view(a, memory);
  const int i = x0 + lane;
  if (i >= nmut || !sched_index_ok(a.status, i < a.J, SCHED_CHK_LIST)) return;
  const int m = v.mut[set * a.J + i], jc = m & 0x7FFF;
  if (!sched_index_ok(a.status, jc < a.J, SCHED_CHK_LIST)) return;
  const int j = v.act[jc];
  const Record rec = load_record(rec_row(a, (w.init || (m >> 15) ? w.src[1] : w.src[0]) + (w.init ? j : jc)));
  uint2 st;
  if (i < stash_rows(a.J)) st = v.stash[set * stash_rows(a.J) + i];
  else st = choices_of(a, draw_one(a.key.k0, round, (uint32_t)j, w.c, w.gen, w.init ? SLOT_INIT : SLOT_MUTATE), j);
  bool slow = rec.w[0] == WIDE;
  if (!slow) {
    uint32_t e[LIST];
#pragma unroll
    for (int k = 0; k < ENTRIES; ++k) e[k] = rec.w[k];
    e[ENTRIES] = NO_NODE;
    int K, N;
    list_totals(e, K, N);
    const uint32_t op = st.y & 3u;
    const int nd = (int)((st.y >> 2) & 0x1FFu), cap_nd = (int)v.cap[nd], k_cap = (int)(st.y >> 16);
    int ns = -1, vs = 0, v_nd = 0;
    const int t = N > 0 ? (int)bounded(st.x, (uint32_t)N) : 0;
#pragma unroll
    for (int k = 0; k < ENTRIES; ++k) {
      if (k == t && N > 0) { ns = entry_node(e[k]); vs = entry_gpus(e[k]); }
      v_nd = entry_node(e[k]) == nd ? entry_gpus(e[k]) : v_nd;
    }
    if (op == 0u || (N > 0 && (op == 1u || nd != ns))) {
      const bool move = op == 2u;
#pragma unroll 1
      for (int q = 0; q < (move ? 2 : 1); ++q)
        list_set(e, op == 1u || q ? ns : nd, q ? 0 : op == 0u ? min(v_nd + 1, cap_nd) : op == 1u ? vs - 1 : min(v_nd + vs, cap_nd));
      list_totals(e, K, N);
    }
    if (K > k_cap || N > a.n_max) {     // replicas above the cap leave from the highest node down, then nodes beyond n_max
      int excess = K - k_cap;
#pragma unroll
      for (int k = LIST - 1; k >= 0; --k) {
        if (e[k] != NO_NODE && excess > 0) {
          const int gpus = entry_gpus(e[k]), take = min(gpus, excess);
          excess -= take;
          e[k] = take == gpus ? NO_NODE : e[k] - (uint32_t)take;
        }
        if (k >= a.n_max) e[k] = NO_NODE;
      }
      list_totals(e, K, N);
    }
    slow = e[ENTRIES] != NO_NODE;
    if (!slow) settle_list<KIND>(a, v, w.dst, jc, e, K, N, true);
  }
  if (slow) {
    const int at = atomicAdd(&v.ctl.nslow, 1);
    if (sched_index_ok(a.status, at < a.J, SCHED_CHK_LIST)) v.wide[a.J - 1 - at] = (uint16_t)m;
  }
}

// As finish_row, for up to 32 of the changed rows.
template <int KIND>
__device__ __noinline__ void finish_lists(const FlowArgs &a, uint32_t memory, int dst, int i0, int nmod, int lane) {
  const FlowView v = flow_view(a, memory);
  if (i0 + lane >= nmod) return;
  const int jc = v.mod[i0 + lane];
  if (v.info[jc] & INFO_WIDE) return;
  const Record rec = load_record(rec_row(a, dst + jc));
  uint32_t e[LIST];
#pragma unroll
  for (int k = 0; k < ENTRIES; ++k) e[k] = entry_gpus(rec.w[k]) == 0 ? NO_NODE : rec.w[k];
  e[ENTRIES] = NO_NODE;
#pragma unroll
  for (int n = ENTRIES - 1; n > 0; --n)
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const uint32_t lo = min(e[k], e[k + 1]);
      e[k + 1] = max(e[k], e[k + 1]);
      e[k] = lo;
    }
  int K, N;
  list_totals(e, K, N);
  settle_list<KIND>(a, v, dst, jc, e, K, N, false);
}

// A wide row that decisions changed, by a warp.
template <int KIND>
__device__ __noinline__ void finish_wide(const FlowArgs &a, uint32_t memory, int dst, int jc, int warp, int lane) {
  const FlowView v = flow_view(a, memory);
  int16_t *dense = v.dense + (size_t)warp * wide_stride(a.NN), *row = wide_row(a, dst + jc);
#pragma unroll 1
  for (int n = lane; n < a.NN; n += 32) dense[n] = __ldcg(row + n);
  __syncwarp();
  int K, N;
  dense_totals(dense, a.NN, lane, K, N);
  const Record out = dense_record(a, dense, v.act[jc], K, N, row, lane);
#pragma unroll
  for (int k = 0; k < REC_WORDS; ++k)
    if (lane == k) put_word<KIND>(a, v, dst, jc, k, out.w[k]);
  if (lane == 0 && N <= ENTRIES) v.info[jc] &= ~INFO_WIDE;
  __syncwarp();
}

// The row pass for wide rows, and for perturbed ones that are or may become wide: a warp each.
template <int KIND>
__device__ __noinline__ void wide_rows(const FlowArgs &a, uint32_t memory, Work w, uint32_t round, int warp, int lane) {
  const FlowView v = flow_view(a, memory);
  const int NN = a.NN, NS = wide_stride(NN), nwide = v.ctl.nwide;
  int16_t *dense = v.dense + (size_t)warp * NS;
#pragma unroll 1
  for (int i = warp; i < nwide + v.ctl.nslow; i += a.warps) {
    const bool slow = i >= nwide;
    const int x = v.wide[slow ? a.J - 1 - (i - nwide) : i], jc = x & 0x7FFF;
    if (!sched_index_ok(a.status, jc < a.J, SCHED_CHK_LIST)) continue;
    const int j = v.act[jc];
    const int from = (x >> 15) || (w.init && slow);
    const Record rec = load_record(rec_row(a, (from ? w.src[1] : w.src[0]) + (w.init ? j : jc)));
    int16_t *const mine = wide_row(a, w.dst + jc);
    if (rec.w[0] == WIDE) {
      const int16_t *contents = wide_source(a, w, from, jc, j);
#pragma unroll 1
      for (int n = lane; n < NS; n += 32) {
        const int16_t e = __ldcg(contents + n);
        dense[n] = e;
        if (!slow) mine[n] = e;
      }
      __syncwarp();
    } else {
      dense_from_list(dense, NS, rec, lane, a.status);
    }
    if (slow) {
      int K, N;
      dense_totals(dense, NN, lane, K, N);
      const u32x4 m = draw_one(a.key.k0, round, (uint32_t)j, w.c, w.gen, w.init ? SLOT_INIT : SLOT_MUTATE);
      const uint32_t op = bounded(m.y, 3u);
      const int nd = (int)bounded(m.w, (uint32_t)NN);
      if (op == 0u) {
        if (lane == 0) dense[nd] = (int16_t)min((int)dense[nd] + 1, (int)v.cap[nd]);
      } else if (N > 0) {
        int ns = nth_occupied(dense, NN, bounded(m.z, (uint32_t)N), lane);
        if (!sched_index_ok(a.status, ns >= 0 && ns < NN && nd < NN, SCHED_CHK_NODE)) ns = nd;
        if (lane == 0 && op == 1u) dense[ns] = (int16_t)(dense[ns] - 1);
        if (lane == 0 && op == 2u && nd != ns) {
          dense[nd] = (int16_t)min((int)dense[nd] + (int)dense[ns], (int)v.cap[nd]);
          dense[ns] = 0;
        }
      }
      __syncwarp();
      dense_totals(dense, NN, lane, K, N);
      dense_caps(dense, NN, K, N, max(0, min(a.k_cap ? a.k_cap[j] : a.k_max, a.k_max)), a.n_max, lane);
      const Record out = dense_record(a, dense, j, K, N, mine, lane);
#pragma unroll
      for (int k = 0; k < REC_WORDS; ++k)
        if (lane == k) put_word<KIND>(a, v, w.dst, jc, k, out.w[k]);
      if (lane == 0) v.info[jc] = (N >= 2 ? INFO_DIST : 0) | (N > ENTRIES ? INFO_WIDE : 0);
      __syncwarp();
    }
    const bool dist = (v.info[jc] & INFO_DIST) != 0, wide = (v.info[jc] & INFO_WIDE) != 0;
    int before = 0;
#pragma unroll 1
    for (int n0 = 0; n0 < NN; n0 += 32) {
      const int n = n0 + lane, e = n < NN ? (int)dense[n] : 0;
      const unsigned m = __ballot_sync(0xffffffffu, e > 0);
      const int k = before + __popc(m & ((1u << lane) - 1u));
      if (e > 0) add_occupant<KIND>(a, v, jc, wide ? 7 : k, ((uint32_t)n << 16) | (uint32_t)e, dist);
      before += __popc(m);
    }
    __syncwarp();
  }
}

// A decision goes straight into the row: entry k of its record (0 GPUs: taken out when the row is
// finished), or its contents.  Decisions of different nodes touch different words.
template <int KIND>
__device__ __forceinline__ void set_entry(const FlowArgs &a, const FlowView &v, int dst, int jc, int k, int n, int gpus) {
  if (!sched_index_ok(a.status, jc < a.J && n < a.NN && (k == 7 || k < ENTRIES), SCHED_CHK_ENTRY)) return;
  const uint32_t e = ((uint32_t)n << 16) | (uint32_t)gpus;
  if (k == 7) wide_row(a, dst + jc)[n] = (int16_t)gpus;
  else if (few(KIND)) v.rec[jc * REC_WORDS + k] = e;
  else rec_row(a, dst + jc)[k] = e;
}

// A row into the list of those that decisions have changed, once.
__device__ __forceinline__ void add_changed(const FlowView &v, int jc, int flag, int J, int *status) {
  // (bytes, so the word around it is updated as a whole)
  const uint32_t bit = (uint32_t)flag << (8 * (jc & 3));
  if ((atomicOr((uint32_t *)v.info + (jc >> 2), bit) & bit) == 0u) {
    const int at = atomicAdd(&v.ctl.nmod, 1);
    if (sched_index_ok(status, at < J, SCHED_CHK_LIST)) v.mod[at] = (uint16_t)jc;
  }
}

// Place of a node in a finished row: of its record, 7: the row is wide.
template <int KIND>
__device__ __forceinline__ int place_of(const FlowArgs &a, const FlowView &v, int dst, int jc, int n) {
  if (v.info[jc] & INFO_WIDE) return 7;
  const Record rec = load_record(rec_row(a, dst + jc));
  int k = 7;
#pragma unroll
  for (int z = 0; z < ENTRIES; ++z) k = entry_node(rec.w[z]) == n ? z : k;
  return k;
}

// Nodes with more occupants than a list holds: the warps walk the column, node by node.  Thread t looks after the
// consecutive rows [t * rpt, (t + 1) * rpt).  Interference: the first distributed occupant in rotated job
// order stays.  Capacity: a prefix sum in job order gives every row the GPUs that come before it in rotated
// order.
template <int KIND>
__device__ __noinline__ void walk_columns(const FlowArgs &a, uint32_t memory, int dst, int set, int JA, int warp, int lane) {
  const FlowView v = flow_view(a, memory);
  const int tid = threadIdx.x, threads = a.warps * 32, J = a.J;
  bar(BAR_ROWS, threads);
  const int rpt = (JA + threads - 1) / threads;
  const int lo = min(JA, tid * rpt), hi = min(JA, lo + rpt);
#pragma unroll 1
  for (int n = 0; n < a.NN; ++n) {
    if (!v.viol[n]) continue;
    const uint32_t rep = v.rep[set * a.NN + n];
    const bool intf = (v.node[2 * n + 1] & 0xFFFFu) >= 2u;
    auto dist = [&](int jc) { return (v.info[jc] & INFO_DIST) != 0; };
    int keep = -1;
    if (intf) {
      int best = 0x7fffffff;
#pragma unroll 1
      for (int jc = lo; jc < hi; ++jc)
        if (dist(jc) && row_at<KIND>(a, dst + jc, n) > 0) {
          int t = (int)v.act[jc] - (int)(rep & 0xFFFFu);
          if (t < 0) t += J;
          best = min(best, t);
        }
      keep = (int)(rep & 0xFFFFu) + block_min(best, v.ctl.red, a.warps);     // the job that stays
      if (keep >= J) keep -= J;
    }
    auto stays = [&](int jc) {
      const int g = row_at<KIND>(a, dst + jc, n);
      return intf && dist(jc) && g > 0 && (int)v.act[jc] != keep ? 0 : g;
    };
    int mine = 0, total;
#pragma unroll 1
    for (int jc = lo; jc < hi; ++jc) mine += stays(jc);
    int running = block_exscan(mine, v.ctl.red, a.warps, total);
    const int excess = total - (int)v.cap[n], o = (int)(rep >> 16);
    int p_o = 0;                          // GPUs of the rows before the offset in job order
    if (excess > 0) {
      if (tid == 0) v.ctl.po = total;     // (no active job at or behind the offset)
      bar(BAR_ROWS, threads);
      int p = running;
#pragma unroll 1
      for (int jc = lo; jc < hi; ++jc) {
        if ((int)v.act[jc] >= o && (jc == 0 || (int)v.act[jc - 1] < o)) v.ctl.po = p;
        p += stays(jc);
      }
      bar(BAR_ROWS, threads);
      p_o = v.ctl.po;
    }
#pragma unroll 1
    for (int jc = lo; jc < hi; ++jc) {
      const int g = row_at<KIND>(a, dst + jc, n), g_eff = stays(jc);
      int take = 0;
      if (excess > 0) {
        const int ahead = (int)v.act[jc] >= o ? running - p_o : total - p_o + running;
        take = min(g_eff, max(excess - ahead, 0));
      }
      running += g_eff;
      v.mod[jc] = g_eff - take == g ? 0 : 1;
      if (g_eff - take != g) {            // into the row
        set_entry<KIND>(a, v, dst, jc, place_of<KIND>(a, v, dst, jc, n), n, g_eff - take);
      }
    }
    bar(BAR_ROWS, threads);
#pragma unroll 1
    for (int i = warp * 4; i < JA; i += a.warps * 4) {
      const int jc = min(i + (lane >> 3), JA - 1);
      const bool live = i + (lane >> 3) < JA && v.mod[jc] && !(v.info[jc] & INFO_WIDE);
      if (__any_sync(0xffffffffu, live)) finish_row<KIND>(a, v, dst, jc, live, warp, lane);
    }
    bar(BAR_ROWS, threads);
#pragma unroll 1
    for (int jc = warp; jc < JA; jc += a.warps)
      if (v.mod[jc] && (v.info[jc] & INFO_WIDE)) finish_wide<KIND>(a, memory, dst, jc, warp, lane);
    bar(BAR_ROWS, threads);
  }
}

// Nodes with more occupants than a group of lanes has: by a warp each, from their lists, and the rows that this
// changes; then the nodes whose lists are too short.  Behind the other nodes' rows, so that a generation without such
// nodes does not have it on its way.
template <int KIND>
__device__ __noinline__ void crowded_nodes(const FlowArgs &a, uint32_t memory, int dst, int set, int JA, int warp, int lane) {
  const FlowView v = flow_view(a, memory);
  const int threads = a.warps * 32;
  bar(BAR_ROWS, threads);                     // (the rows of the other nodes are finished)
  if (threadIdx.x == 0) v.ctl.nmod = 0;
  bar(BAR_ROWS, threads);
#pragma unroll 1
  for (int n = warp; n < a.NN; n += a.warps) {
    if (!v.viol[n]) continue;
    const uint2 here = ((const uint2 *)v.node)[n];
    const int count = (int)(here.y >> 16);
    if (count > FLOW_OCC + a.more) {
      if (lane == 0) v.ctl.walk = 2;
      continue;
    }
    const uint32_t rep = v.rep[set * a.NN + n];
    auto list = [&](int i) { return i < FLOW_OCC ? v.occ[n * FLOW_OCC + i] : v.more[n * a.more + i - FLOW_OCC]; };
    auto gpus = [&](uint32_t e) { return (int)((e >> 13) & 0x7FFu); };
    auto place = [&](uint32_t e, uint32_t offset) {
      const int jc = (int)(e & 0x1FFFu), r = (sched_index_ok(a.status, jc < a.J, SCHED_CHK_LIST) ? (int)v.act[jc] : 0) - (int)offset;
      return r < 0 ? r + a.J : r;
    };
    auto rot_i = [&](uint32_t e) { return place(e, rep & 0xFFFFu); };
    auto rot_c = [&](uint32_t e) { return place(e, rep >> 16); };
    const CrowdPlaces at = crowd_places(list, count, a.J, (int)here.x, (here.y & 0xFFFFu) >= 2u, (int)v.cap[n], lane, gpus, rot_i, rot_c);
#pragma unroll 1
    for (int i = lane; i < count; i += 32) {
      const uint32_t e = list(i);
      const int jc = (int)(e & 0x1FFFu), keeps = at.keeps(e, gpus(e), rot_i(e), rot_c(e));
      if (keeps == gpus(e)) continue;
      set_entry<KIND>(a, v, dst, jc, place_of<KIND>(a, v, dst, jc, n), n, keeps);
      add_changed(v, jc, INFO_AGAIN, a.J, a.status);
    }
    __syncwarp();
    if (lane == 0) v.viol[n] = 0;
  }
  bar(BAR_ROWS, threads);
  const int nmod = v.ctl.nmod;
#pragma unroll 1
  for (int i0 = warp * 4; i0 < nmod; i0 += a.warps * 4) {
    const int jc = v.mod[min(i0 + (lane >> 3), nmod - 1)];
    finish_row<KIND>(a, v, dst, jc, i0 + (lane >> 3) < nmod && !(v.info[jc] & INFO_WIDE), warp, lane);
  }
  bar(BAR_ROWS, threads);                     // (a wide one may turn into a record: not to be taken for one above)
#pragma unroll 1
  for (int i = warp; i < nmod; i += a.warps) {
    const int jc = v.mod[i];
    if (v.info[jc] & INFO_WIDE) finish_wide<KIND>(a, memory, dst, jc, warp, lane);
  }
  if (v.ctl.walk == 2) walk_columns<KIND>(a, memory, dst, set, JA, warp, lane);
}

// An elite child: the records (and contents) of the candidate of its rank, as they are.
template <int KIND>
__device__ __noinline__ void copy_candidate(const FlowArgs &a, int from, int to, int rows) {
#pragma unroll 4
  for (int i = threadIdx.x; i < rows; i += a.warps * 32) {
    const Record r = load_record(rec_row(a, from + i));
    store_record(rec_row(a, to + i), r);
    if (r.w[0] == WIDE) {
#pragma unroll 1
      for (int v = 0; v < wide_stride(a.NN) / 8; ++v)
        ((uint4 *)wide_row(a, to + i))[v] = __ldcg((const uint4 *)wide_row(a, from + i) + v);
    }
  }
}

// Two calls that differ in their slot, a round at a time: a twelfth of the code of draw_two for half again its instructions.
// A small round's blocks have issue slots to spare and no room for code: what all its warps go through in a
// generation should stay in the SM's instruction cache.
__device__ __forceinline__ void draw_two_rolled(uint32_t k0, uint32_t k1, uint32_t idx, uint32_t cand, uint32_t gen, uint32_t slot_a,
                                                uint32_t slot_b, uint32_t &a_x, u32x4 &b) {
  u32x4 x = {idx, cand, gen, slot_a}, y = {idx, cand, gen, slot_b};
#pragma unroll 1
  for (int r = 0; r < 10; ++r) {
    x = philox_round(x, k0, k1);
    y = philox_round(y, k0, k1);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  a_x = x.x;
  b = y;
}

// The warps that draw: a candidate's random numbers of a step (each row's parent and whether it is perturbed, the
// perturbed rows' list, the nodes' offsets).  Nothing in it waits for another block, so it is done while the
// item before is worked on; the block's barrier hands it over.
template <int KIND>
__device__ __noinline__ void draw_items(const FlowArgs &a, uint32_t memory, uint32_t round, int JA) {
  const FlowView v = flow_view(a, memory);
  const int J = a.J, NN = a.NN, P = a.P, lane = threadIdx.x & 31;
  const int D = (int)blockDim.x - a.warps * 32, d = (int)threadIdx.x - a.warps * 32;
  int set = 0;
  uint32_t c = blockIdx.x;
#pragma unroll 1
  for (int s = 0; s <= a.generations; set ^= 1) {
    const bool init = s == 0;
    const uint32_t gen = (uint32_t)(s - 1);                 // (GEN_INIT is -1)
    const uint32_t c_next = c + gridDim.x < (uint32_t)P ? c + gridDim.x : blockIdx.x;
    const int s_next = c_next > c ? s : s + 1;
    // the candidates of the next item's tournaments: looked at before the barrier that hands that item over
    if (d < 32 && s_next > 0) {
      u32x4 sel;
      uint32_t unused;
      if (few(KIND)) draw_two_rolled(a.key.k0, round, 0u, c_next, (uint32_t)(s_next - 1), SLOT_SELECT, SLOT_SELECT, unused, sel);
      else sel = draw_one(a.key.k0, round, 0u, c_next, (uint32_t)(s_next - 1), SLOT_SELECT);
      if (lane < 4) v.ctl.sel[set ^ 1][lane] = bounded(lane == 0 ? sel.x : lane == 1 ? sel.y : lane == 2 ? sel.z : sel.w, (uint32_t)P);
    }
    if (init || (int)c >= a.num_elite) {
#pragma unroll 1
      for (int i = d; i < JA + NN; i += D) {
        const bool row = i < JA;
        const int jc = row ? i : 0;
        const uint32_t idx = row ? v.act[jc] : (uint32_t)(i - JA);
        u32x4 m;
        uint32_t x = 0u;
        const uint32_t slot_a = row ? SLOT_XOVER : SLOT_REPAIR_INTF, slot_b = !row ? SLOT_REPAIR_CAP : init ? SLOT_INIT : SLOT_MUTATE;
        if (few(KIND)) draw_two_rolled(a.key.k0, round, idx, c, gen, slot_a, slot_b, x, m);
        else draw_two(a.key.k0, round, idx, c, gen, slot_a, slot_b, x, m);
        if (!row) {
          v.rep[set * NN + (int)idx] = bounded(x, (uint32_t)J) | (bounded(m.x, (uint32_t)J) << 16);
          continue;
        }
        const bool sec = !init && (x >> 31) != 0u, mut = init ? c > 0u && m.x < a.thr_init : m.x < a.thr_mutate;
        v.flag[set * J + jc] = (sec ? 1 : 0) | (mut ? 2 : 0);
        if (mut) {
          const int at = atomicAdd(&v.ctl.nmut[set], 1);
          if (!sched_index_ok(a.status, at < J, SCHED_CHK_LIST)) continue;
          v.mut[set * J + at] = (uint16_t)(jc | (sec ? 0x8000 : 0));
          if (at < stash_rows(J))
            v.stash[set * stash_rows(J) + at] = choices_of(a, m, (int)idx);
        }
      }
    }
    __syncthreads();
    if (!v.ctl.hand[set].z) return;
    c = c_next;
    s = s_next;
  }
}

template <int KIND>
__global__ void __launch_bounds__(kind_threads(KIND), kind_blocks(KIND)) flow_kernel(const __grid_constant__ FlowArgs a) {
  extern __shared__ __align__(16) unsigned char flow_memory[];
  const uint32_t memory = (uint32_t)__cvta_generic_to_shared(flow_memory);
  const FlowView v = flow_view(a, memory);
  const int J = a.J, NN = a.NN, P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = a.warps;

  const uint32_t round = __ldg(a.key.round_ptr), base = __ldg(a.r.base);
  const int JA = *a.r.num_act;
#pragma unroll 1
  for (int i = tid; i < JA; i += blockDim.x) v.act[i] = a.r.act[i];
#pragma unroll 1
  for (int i = tid; i < J; i += blockDim.x) v.term[i] = 0.f;
#pragma unroll 1
  for (int i = tid; i < a.chunks * 8; i += blockDim.x) v.sums[i] = 0.0;
#pragma unroll 1
  for (int i = tid; i < NN; i += blockDim.x) {
    v.cap[i] = (int16_t)max((int)a.cap[i], 0);
    if (a.rack) v.rack[i] = a.rack[i];
    v.node[2 * i] = v.node[2 * i + 1] = 0u;
    v.viol[i] = 0;
  }
  if (tid == 0) {
    FlowCtl &c = v.ctl;
    c.nmut[0] = c.nmut[1] = c.nwide = c.nslow = c.nmod = c.walk = 0;
    c.hand[0] = c.hand[1] = make_int4(0, 0, 1, 0);
  }
  __syncthreads();
  if (few(KIND)) {
#pragma unroll 1
    for (int i = tid; i < JA * REC_WORDS; i += blockDim.x)
      v.same[i] = __ldg(a.r.same + (size_t)v.act[i / REC_WORDS] * REC_WORDS + (i & (REC_WORDS - 1)));
    if (a.at.terms >= 0) {
      const int row = a.classes * (a.k_max + 1);
#pragma unroll 1
      for (int i = warp; i < JA; i += (int)(blockDim.x >> 5))
#pragma unroll 4
        for (int x = lane; x < row; x += 32) v.terms[i * row + x] = __ldg(a.r.terms + (size_t)v.act[i] * row + x);
    }
  }
  if (warp >= W) {
    draw_items<KIND>(a, memory, round, JA);
    return;
  }

  const int threads = W * 32, g = lane >> 3, nv = (min(J, SUM_THREADS) + 31) >> 5;
  const bool last_warp = warp == W - 1;
  const int PJ = P * J, cur_rows = (int)((a.r.cur_rec - a.r.rec) / REC_WORDS);
  auto pub_of = [&](int step, uint32_t cand) { return a.r.pub + ((size_t)(step & (DEPTH - 1)) * P + cand) * PUB_STRIDE; };
  // Items: this block's candidates of step 0 (the initial population), of step 1 (generation 0), ...
  int s = 0, set = 0;
  Work w;
  w.c = blockIdx.x;
#pragma unroll 1
  while (s <= a.generations) {
    const uint32_t c = w.c;
    const bool init = s == 0, elite = !init && (int)c < a.num_elite;
    w.init = init;
    w.gen = (uint32_t)(s - 1);
    w.dst = (s & (DEPTH - 1)) * PJ + (int)c * J;

    // ---- parents ----------------------------------------------------------------------------------
    // The candidate of its rank for an elite child (which needs every key), else the better-ranked of
    // two random pairs (which needs four).  Candidate 0 waits for every key in any case: that it has
    // published step t tells everybody that nobody reads step t - 2 any more.
    if (!init && (elite || c == 0u)) {
      bool ok = true;
#pragma unroll 1
      for (int i = tid; i < P && ok; i += threads) {
        const unsigned long long word = wait_tag(pub_of(s - 1, i), base + (uint32_t)(s - 1), a.wait_limit, a.status);
        ok = word != 0ull;
        v.keys[i] = (uint32_t)word;
      }
      waited();
      if (!ok) v.ctl.hand[set].z = 0;
      bar(BAR_ROWS, threads);
    }
    if (last_warp) {
      // (initial population: an unperturbed row is the current allocation's after the row caps, a perturbed one
      // starts from it before them; rows of the current allocation lie by job)
      const int before = init ? cur_rows : ((s - 1) & (DEPTH - 1)) * PJ;
      int parent = init ? lane >> 1 : 0;
      if (!init) {
        unsigned long long word = 1ull;
        const uint32_t mine = v.ctl.sel[set][lane & 3], other = __shfl_down_sync(0xffffffffu, mine, 1);
        const unsigned long long *const watched = lane == 4 ? pub_of(s - 2, 0u) : pub_of(s - 1, mine);
        const uint32_t tag = base + (uint32_t)(lane == 4 ? s - 2 : s - 1);
        if (lane == 4 ? s >= DEPTH : lane < 4 && !elite) word = wait_tag(watched, tag, a.wait_limit, a.status);
        waited();
        const uint32_t key = (uint32_t)word, ko = __shfl_down_sync(0xffffffffu, key, 1);
        parent = tournament_winner(key, (int)mine, ko, (int)other);
        if (word == 0ull) v.ctl.hand[set].z = 0;
        if (elite) parent = v.ctl.hand[set].z ? candidate_of_rank(v.keys, P, (int)c, (uint16_t *)(v.keys + P), lane) : 0;
        if (!sched_index_ok(a.status, parent >= 0 && parent < P, SCHED_CHK_SLOT)) parent = 0;
      }
      if (lane == 0) v.ctl.hand[set].x = before + parent * J;
      if (lane == 2) v.ctl.hand[set].y = before + parent * J;
      if (elite && lane == 0) v.ctl.hand[set].w = parent;
    }
    __syncthreads();
    const int4 hand = v.ctl.hand[set];
    if (!hand.z) return;                      // (a wait ran out: the status says so)
    w.src[0] = hand.x;
    w.src[1] = hand.y;

    auto next_item = [&]() {
      set ^= 1;
      w.c += gridDim.x;
      if (w.c >= (uint32_t)P) { w.c = blockIdx.x; ++s; }
    };
    if (elite) {
      const uint32_t key = v.keys[hand.w];
      copy_candidate<KIND>(a, w.src[0], w.dst, JA);
      bar(BAR_ROWS, threads);
      if (tid == 0) {
        publish(pub_of(s, c), base + (uint32_t)s, key);
        if (s == a.generations) a.fitness[c] = __uint_as_float(key ^ ((key >> 31) ? 0x80000000u : 0xFFFFFFFFu));
      }
      next_item();
      continue;
    }

    // ---- the rows: perturbed ones (from the last warp on) and the others --------------------------------
    const uint8_t *const flag = v.flag + set * J;
    auto note_wide = [&](int jc, uint32_t f) {
      const int at = atomicAdd(&v.ctl.nwide, 1);
      if (sched_index_ok(a.status, at < J, SCHED_CHK_LIST)) v.wide[at] = (uint16_t)(jc | ((f & 1u) ? 0x8000 : 0));
      v.info[jc] = INFO_DIST | INFO_WIDE;
    };
    const int nmut = v.ctl.nmut[set];
#pragma unroll 1
    for (int x = (W - 1 - warp) * 4; x < nmut && !(!few(KIND) && nmut > LISTS_FROM * W); x += W * 4)
      perturb_rows<KIND>(a, v, w, round, set, x, nmut, warp, lane);
    if constexpr (!few(KIND))
      if (nmut > LISTS_FROM * W)
#pragma unroll 1
        for (int x = (W - 1 - warp) * 32; x < nmut; x += W * 32) perturb_lists<KIND>(a, memory, w, round, set, x, nmut, lane);
    constexpr int RB = shape_of(KIND) == SOME_ALONE || !few(KIND) ? 2 : 1;       // rows of a thread whose loads travel together
#pragma unroll 1
    for (int jc0 = tid; jc0 < JA; jc0 += RB * threads) {
      Record rec[RB];
      uint32_t f[RB];
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        const int jc = min(jc0 + q * threads, JA - 1);
        f[q] = jc0 + q * threads < JA ? (uint32_t)flag[jc] : 2u;
        rec[q] = load_record(rec_row(a, ((f[q] & 1u) ? w.src[1] : w.src[0]) + (init ? (int)v.act[jc] : jc)));
      }
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        const int jc = jc0 + q * threads;
        if (f[q] & 2u) continue;
        store_record(rec_row(a, w.dst + jc), rec[q]);
        if (few(KIND)) {
          ((uint4 *)v.rec)[2 * jc] = make_uint4(rec[q].w[0], rec[q].w[1], rec[q].w[2], rec[q].w[3]);
          ((uint4 *)v.rec)[2 * jc + 1] = make_uint4(rec[q].w[4], rec[q].w[5], rec[q].w[6], rec[q].w[7]);
        }
        v.term[v.act[jc]] = __uint_as_float(rec[q].w[REC_TERM]);
        if (rec[q].w[0] == WIDE) {
          note_wide(jc, f[q]);
          continue;
        }
        const bool dist = rec[q].w[1] != NO_NODE;
        v.info[jc] = dist ? INFO_DIST : 0;
        if (rec[q].w[0] != NO_NODE) add_occupant<KIND>(a, v, jc, 0, rec[q].w[0], dist);
#pragma unroll 1
        for (int x = 1; x < ENTRIES; ++x) {           // (few rows have more: one copy of the code)
          uint32_t e = rec[q].w[1];
#pragma unroll
          for (int z = 2; z < ENTRIES; ++z) e = z == x ? rec[q].w[z] : e;
          if (e == NO_NODE) break;
          add_occupant<KIND>(a, v, jc, x, e, dist);
        }
      }
    }
    bar(BAR_ROWS, threads);
    const bool any_wide = (v.ctl.nwide | v.ctl.nslow) != 0;
    if (any_wide) {
      wide_rows<KIND>(a, memory, w, round, warp, lane);
      bar(BAR_ROWS, threads);
    }

    // ---- node decisions: a lane looks at a node, groups of 16 lanes decide the nodes that hold two
    // distributed jobs or more GPUs than they have; nodes are dealt out round robin, so that violations
    // spread over the warps ---------------------------------------------------------------------------
#pragma unroll 1
    for (int n0 = warp; n0 < NN; n0 += 32 * W) {
      const int n_l = n0 + lane * W;
      bool bad = false;
      if (n_l < NN) {
        const uint2 here = ((const uint2 *)v.node)[n_l];
        bad = (here.y & 0xFFFFu) >= 2u || (int)here.x > (int)v.cap[n_l];
      }
      unsigned todo = __ballot_sync(0xffffffffu, bad);
#pragma unroll 1
      while (todo) {
        const int b0 = __ffs(todo) - 1;
        todo &= todo - 1;
        const int b1 = __ffs(todo) - 1;       // (-1: there is none)
        todo &= todo - 1;
        const int b = (lane & 16) ? b1 : b0, sub = lane & 15;
        const int n = n0 + max(b, 0) * W;
        const uint2 here = ((const uint2 *)v.node)[n];
        const uint32_t rep = v.rep[set * NN + n], e = v.occ[n * FLOW_OCC + sub];
        const int count = b >= 0 ? (int)(here.y >> 16) : 0, cap_n = (int)v.cap[n];
        const bool listed = count <= FLOW_OCC, have = listed && sub < count;   // else: below
        const int jc = have ? (int)(e & 0x1FFFu) : 0, had = have ? (int)((e >> 13) & 0x7FFu) : 0;
        const int j = sched_index_ok(a.status, jc < JA, SCHED_CHK_LIST) ? (int)v.act[jc] : 0;
        int ri = j - (int)(rep & 0xFFFFu), rc = j - (int)(rep >> 16);
        if (ri < 0) ri += J;
        if (rc < 0) rc += J;
        const int most = max(__shfl_sync(0xffffffffu, count, 0), __shfl_sync(0xffffffffu, count, 16));
        const int keeps = decide(had, (e >> 31) != 0u, have, min(most, FLOW_OCC), (here.y & 0xFFFFu) >= 2u, (int)here.x, cap_n, ri, rc);
        if (have && keeps != had) {
          set_entry<KIND>(a, v, w.dst, jc, (int)((e >> 25) & 7u), n, keeps);
          add_changed(v, jc, INFO_CHANGED, J, a.status);
        }
        if (b >= 0 && sub == 0 && !listed) { v.viol[n] = 1; v.ctl.walk = 1; }
        __syncwarp();
      }
    }
    bar(BAR_ROWS, threads);

    // ---- rows the decisions change, then columns that have to be walked --------------------------------
    const int nmod = v.ctl.nmod, walk = v.ctl.walk;
#pragma unroll 1
    for (int i0 = warp * 4; i0 < nmod && !(!few(KIND) && nmod > LISTS_FROM * W); i0 += W * 4) {
      const int jc = v.mod[min(i0 + g, nmod - 1)];
      finish_row<KIND>(a, v, w.dst, jc, i0 + g < nmod && !(v.info[jc] & INFO_WIDE), warp, lane);
    }
    if constexpr (!few(KIND))
      if (nmod > LISTS_FROM * W)
#pragma unroll 1
        for (int i0 = warp * 32; i0 < nmod; i0 += W * 32) finish_lists<KIND>(a, memory, w.dst, i0, nmod, lane);
    if (any_wide) {                           // wide rows among them
      bar(BAR_ROWS, threads);                 // (one may turn into a record here: not to be taken for one above)
#pragma unroll 1
      for (int i = warp; i < nmod; i += W) {
        const int jc = v.mod[i];
        if (v.info[jc] & INFO_WIDE) finish_wide<KIND>(a, memory, w.dst, jc, warp, lane);
      }
    }
    if (walk && (KIND & CROWDED)) crowded_nodes<KIND>(a, memory, w.dst, set, JA, warp, lane);
    else if (walk) walk_columns<KIND>(a, memory, w.dst, set, JA, warp, lane);
    bar(BAR_ROWS, threads);

    // ---- fitness (Eq. 14) from the rows' terms, in the order of the dense kernel: per chunk of rows, thread
    // t adds rows t, t + 256, ... in double, a shuffle tree per warp, the warps in index order; then the
    // chunks in index order.  Meanwhile the last warp makes everybody's rows visible to the other blocks; then it
    // publishes. -----------------------------------------------------------------------------------------
    if (last_warp) {
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      bar(BAR_KEY, 64);
      if (lane == 0) {
        const unsigned long long word = v.ctl.word;
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(pub_of(s, c)), "l"(word) : "memory");   // (behind this thread's fence)
      }
    } else {
      constexpr bool ONE = shape_of(KIND) == FEW_ALONE;     // (up to 256 rows: one chunk, a row a thread)
      const int chunks = ONE ? 1 : a.chunks;
#pragma unroll 1
      for (int x = warp; x < chunks * nv; x += W - 1) {
        const int ch = ONE || chunks == 1 ? 0 : x / nv, vw = x - ch * nv;
        double acc = 0.0;
        if (ONE) {
          if (vw * 32 + lane < J) acc = (double)v.term[vw * 32 + lane];
        } else {
          const int j0 = ch * a.rows_per_chunk, j1 = min(J, j0 + a.rows_per_chunk);
#pragma unroll 1
          for (int j = j0 + vw * 32 + lane; j < j1; j += SUM_THREADS) acc += (double)v.term[j];
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) v.sums[ch * 8 + vw] = acc;
      }
      if (chunks * nv > 1) bar(BAR_SUMS, threads - 32);
      if (warp == 0) {
        if (lane == 0) {
          double sum = 0.0;
#pragma unroll 1
          for (int ch = 0; ch < chunks; ++ch) {
            double part[8], t = 0.0;            // (warps that do not exist left zeros)
#pragma unroll
            for (int x = 0; x < 8; ++x) part[x] = v.sums[ch * 8 + x];
#pragma unroll
            for (int x = 0; x < 8; ++x) t += part[x];
            sum += t;
          }
          const float f = fitness_finalise(a.tp.mode, a.tp.p, sum, (double)JA);
          v.ctl.word = ((unsigned long long)(base + (uint32_t)s) << 32) | order_key(__float_as_uint(f));
          if (s == a.generations) a.fitness[c] = f;
        }
        __syncwarp();
        bar(BAR_KEY, 64);
      }
      // for the next candidate
#pragma unroll 1
      for (int i = threads - 33 - tid; i < NN; i += threads - 32) {
        ((uint2 *)v.node)[i] = make_uint2(0u, 0u);
        v.viol[i] = 0;
      }
      if (tid == threads - 33) { v.ctl.nmut[set] = 0; v.ctl.nwide = 0; v.ctl.nslow = 0; v.ctl.nmod = 0; v.ctl.walk = 0; }
    }
    next_item();
  }
}

// The best candidate (largest key, lowest index on ties) and its rows as a dense matrix; the next
// round's tags begin behind this round's.
__global__ void __launch_bounds__(256) flow_finish_kernel(FlowArgs a) {
  __shared__ unsigned long long s_best[8];
  __shared__ uint16_t s_place[FLOW_MAX_JOBS];      // place of a job's row, 0xFFFF: the job is not active
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, P = a.P, J = a.J, NN = a.NN, NS = wide_stride(NN);
  asm volatile("griddepcontrol.wait;" ::: "memory");
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

}  // namespace

namespace {

// The pieces of the round's one allocation (tables and fitness among them); total with base NULL.
struct FlowArena {
  FlowRows r;
  float *goodput, *speedup, *speedup_rack, *fitness;
  size_t total;
};

int flow_classes(const sched_ctx *ctx) { return ctx->d_rack ? 3 : 2; }

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
  TAKE(r.terms, float, J * flow_classes(ctx) * ctx->KD * 4);
  TAKE(r.pen, float, J * 4);
  TAKE(r.act, uint16_t, J * 2);
  TAKE(r.num_act, int, 4);
  TAKE(r.base, uint32_t, 4);
  TAKE(r.pub, unsigned long long, DEPTH * P * PUB_STRIDE * 8);
  TAKE(r.cur_wide, int16_t, 2 * J * NS * 2);
  TAKE(r.rec, uint32_t, DEPTH * P * J * REC_WORDS * 4);
  TAKE(r.wide, int16_t, DEPTH * P * J * NS * 2);
#undef TAKE
  f.total = off;
  return f;
}

FlowSmem flow_smem(const sched_ctx *ctx, int kind, int warps, bool terms, int more) {
  const sched_config &c = ctx->cfg;
  const int J = c.num_jobs, NN = c.num_nodes, P = c.population;
  int rows, chunks, off = 0;
  fitness_chunking(ctx, P, rows, chunks);
  FlowSmem L;
  auto take = [&](size_t bytes) {
    const int at = off;
    off += (int)((bytes + 15) & ~(size_t)15);
    return at;
  };
  take(sizeof(FlowCtl));
  L.act = take((size_t)J * 2);
  L.term = take((size_t)J * 4);
  L.info = take((size_t)J);
  L.node = take((size_t)NN * 8);
  L.occ = take((size_t)NN * FLOW_OCC * 4);
  L.more = take((size_t)NN * more * 4);
  L.viol = take((size_t)NN);
  L.cap = take((size_t)NN * 2);
  L.rack = take(ctx->d_rack ? (size_t)NN * 2 : 0);
  L.mut = take(2 * (size_t)J * 2);
  L.mod = take((size_t)J * 2);
  L.stash = take(2 * (size_t)stash_rows(J) * 8);
  L.flag = take(2 * (size_t)J);
  L.dense = take((size_t)warps * wide_stride(NN) * 2);
  L.rep = take(2 * (size_t)NN * 4);
  L.keys = take((size_t)P * 6);      // and a list of candidates behind them
  L.sums = take((size_t)chunks * 8 * 8);
  L.scratch = take((size_t)warps * 32 * 4);
  L.rec = few(kind) ? take((size_t)J * REC_WORDS * 4) : 0;
  L.same = few(kind) ? take((size_t)J * REC_WORDS * 4) : 0;
  L.terms = terms ? take((size_t)J * flow_classes(ctx) * ctx->KD * 4) : -1;
  L.total = off;
  return L;
}

int flow_kind(const sched_ctx *ctx) {
  const int J = ctx->cfg.num_jobs, NN = ctx->cfg.num_nodes, P = ctx->cfg.population;
  const bool alone = P <= ctx->num_sms, two = P <= 2 * ctx->num_sms;
  if (J <= SMEM_RECORDS) return alone ? FEW_ALONE : FEW;
  if (alone && flow_smem(ctx, SOME_ALONE, SOME_WARPS, false, 0).total <= FLOW_MAX_SMEM) return SOME_ALONE;
  if (two && 79 * J + 115 * NN + 6 * P <= 96 * 1024) return FEW;        // (what two blocks find room for on an SM)
  return two || J > MANY_TWO_JOBS ? MANY_TWO : MANY;
}

// The launch's shape.
struct FlowShape {
  int warps, draw_warps, blocks, more;
  FlowSmem at;
};

using FlowKernel = void (*)(FlowArgs);
FlowKernel flow_kernel_for(const sched_ctx *ctx, bool crowded) {
  switch (flow_kind(ctx) | (crowded ? CROWDED : 0)) {
    case FEW_ALONE: return flow_kernel<FEW_ALONE>;
    case SOME_ALONE: return flow_kernel<SOME_ALONE>;
    case FEW: return flow_kernel<FEW>;
    case MANY: return flow_kernel<MANY>;
    case MANY_TWO: return flow_kernel<MANY_TWO>;
    case FEW_ALONE | CROWDED: return flow_kernel<FEW_ALONE | CROWDED>;
    case SOME_ALONE | CROWDED: return flow_kernel<SOME_ALONE | CROWDED>;
    case FEW | CROWDED: return flow_kernel<FEW | CROWDED>;
    case MANY | CROWDED: return flow_kernel<MANY | CROWDED>;
    default: return flow_kernel<MANY_TWO | CROWDED>;
  }
}

// What a node's list should hold beyond FLOW_OCC occupants, by the rows that a step (the initial population, too)
// perturbs, in at most 16 KB.  A node with more than its list holds is walked, row by row, by the whole block.  60
// generations with lists of 16 and with these (us): a fifth of the rows perturbed, 8 nodes x 1024 jobs x 300 candidates
// 6435 -> 1679, 16 x 1024 x 512 2729 -> 1840, 4 x 300 x 512 1083 -> 773; a fiftieth, but three of ten at first, 4 x 1024 x 512
// 1032 -> 870, 8 x 512 x 148 388 -> 385.  Where crowds are rare they cost up to 2 % (8 x 300 x 297 450 -> 459).
int flow_more(const sched_ctx *ctx) {
  const sched_config &c = ctx->cfg;
  return listed_occupants(ctx, std::max(c.thr_mutate, c.thr_init), 256 * FLOW_OCC / c.num_nodes) - FLOW_OCC;
}

// A block for every candidate if they fit the GPU.  Warps that work on rows and warps that draw, measured.  Before the keys were
// set apart, which took the same off all of them: testbed (48 jobs) 3 + 2 540 us, 4 + 2 513, 6 + 2 508, 8 + 2 and 8 + 4 505, 12 + 4
// 509; 96 jobs in racks 662, 621, 557, 547, 542, 542; two blocks an SM (210 jobs) 8 + 2 760, 10 + 3 698, 12 + 3 693; 1024 jobs, four
// blocks an SM 6 + 2 3896, 7 + 2 3700, 7 + 3 3774, 8 + 2 3740.  Since, 30 generations: MANY_TWO, 148 candidates x 4000 jobs 10 + 3
// 1563, 12 + 2 2143, 12 + 4 1373, 14 + 2 2137; SOME_ALONE, 64 x 1100 12 + 4 694, 14 + 6 647, 16 + 2 918, 16 + 4 642, 64 x 2000 821,
// 759, 1391, 806 (with so many rows the draws are what takes long); FEW, 54 jobs x 600 candidates 6 + 2 in two turns 628, 4 + 2
// 447, 4 + 1 452, 3 + 1 487; x 888 703, 770, 533, 588; x 1100 753, 827, 902, 675; x 1300 in three, two, two and two turns 1040, 882,
// 956, 1073.  The terms' table finds room in shared memory where that does not cost a block its place.
FlowShape flow_shape(const sched_ctx *ctx) {
  const sched_config &c = ctx->cfg;
  const int kind = flow_kind(ctx);
  FlowShape best = {};
  int warps, draw;
  switch (kind) {
    case MANY: warps = 7; draw = 2; break;
    case MANY_TWO: warps = 12; draw = 4; break;
    case SOME_ALONE: warps = SOME_WARPS; draw = 4; break;
    case FEW_ALONE: warps = 8; draw = 4; break;
    default: {
      // up to eight blocks an SM, and no more turns than that takes; then as few blocks an SM as the turns leave
      const int most = std::max(1, std::min(8, 227 * 1024 / (flow_smem(ctx, kind, 3, false, 0).total + 1024)));
      const int turns = (c.population + most * ctx->num_sms - 1) / (most * ctx->num_sms);
      const int per_sm = (c.population + turns * ctx->num_sms - 1) / (turns * ctx->num_sms);
      warps = per_sm <= 2 ? 12 : per_sm == 3 ? 8 : per_sm == 4 ? 6 : per_sm <= 6 ? 4 : 3;
      draw = per_sm <= 2 ? 3 : per_sm <= 5 ? 2 : 1;
    }
  }
  for (int x = few(kind) ? 3 : 1; x >= 0 && best.blocks < c.population; --x) {      // terms and long lists, terms, long lists, neither
    const bool terms = (x & 2) != 0;
    const int more = (x & 1) ? flow_more(ctx) : 0;
    if ((x & 1) && more == 0) continue;
    FlowShape f = {warps, draw, 0, more, flow_smem(ctx, kind, warps, terms, more)};
    const FlowKernel kernel = flow_kernel_for(ctx, more > 0);
    int fit = 0;
    if (f.at.total > FLOW_MAX_SMEM ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FLOW_MAX_SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, (warps + draw) * 32, f.at.total) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    f.blocks = std::min(c.population, fit * ctx->num_sms);
    if (f.blocks > best.blocks) best = f;
  }
  return best;
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
  if ((long long)(DEPTH + 1) * c.population * c.num_jobs >= 1ll << 31) return SCHED_OK;      // (rows are counted in 32 bits)
  int coop = 0, blocks = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess || !coop) {
    cudaGetLastError();
    return SCHED_OK;
  }
  const FlowShape shape = flow_shape(ctx);
  blocks = shape.blocks;
  if (blocks < 1) return SCHED_OK;
  ctx->fl_warps = shape.warps;
  ctx->fl_draw_warps = shape.draw_warps;
  ctx->fl_terms = shape.at.terms >= 0;
  ctx->fl_more = shape.more;
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
  // no tag matches before it is published.  (Records are not cleared: a round reads those of candidates that have published
  // theirs, at places below the number of active jobs, and all of these are written before that.)
  SCHED_CUDA_CHECK(ctx, cudaMemsetAsync(f.r.pub, 0, DEPTH * (size_t)c.population * PUB_STRIDE * 8, ctx->stream));
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
  a.num_elite = c.num_elite; 
  a.nmin = ctx->d_nmin; a.classes = flow_classes(ctx);
  a.thr_init = c.thr_init; a.thr_mutate = c.thr_mutate;
  a.key = make_key(c.seed, ctx->d_round);
  fitness_chunking(ctx, c.population, a.rows_per_chunk, a.chunks);
  a.fitness = ctx->d_fit;
  a.wait_limit = ctx->fl_wait_limit;
  a.status = ctx->d_status;
  return a;
}

// A launch that may begin while the kernel before it on the stream ends.
static cudaError_t launch_beside(sched_ctx *ctx, FlowKernel kernel, int blocks, int threads, const FlowArgs &a) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)blocks);
  lc.blockDim = dim3((unsigned)threads);
  lc.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kernel, a);
}

// The search of a round, after its tables.
int launch_round_flow(sched_ctx *ctx, const sched_jobs *jobs, const int16_t *d_cur, int32_t generations, int16_t *d_best,
                      float *d_best_fitness) {
  const sched_config &c = ctx->cfg;
  FlowArgs a = flow_args(ctx, jobs, d_cur);
  a.generations = generations;
  a.warps = ctx->fl_warps;
  a.more = ctx->fl_more;
  const bool terms = ctx->fl_terms && (generations > TERMS_FROM || (c.num_jobs <= TERMS_JOBS && generations >= c.num_jobs));
  a.at = flow_smem(ctx, flow_kind(ctx), ctx->fl_warps, terms, ctx->fl_more);
  a.best = d_best; a.best_fitness = d_best_fitness;
  {
    TimedLaunch tl_(ctx, KK_FLOW_BUILD);
    // (beside the tables' last kernel: what needs no table is done while that still writes)
    SCHED_CUDA_CHECK(ctx, launch_beside(ctx, flow_build_kernel, (c.num_jobs + 3) / 4, 128, a));
  }
  SCHED_LAUNCH_CHECK(ctx);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)ctx->fl_blocks);
  lc.blockDim = dim3((unsigned)(ctx->fl_warps + ctx->fl_draw_warps) * 32);
  lc.dynamicSmemBytes = (size_t)a.at.total;
  lc.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  {
    TimedLaunch tl_(ctx, KK_FLOW);
    SCHED_CUDA_CHECK(ctx, cudaLaunchKernelEx(&lc, flow_kernel_for(ctx, ctx->fl_more > 0), a));
  }
  SCHED_LAUNCH_CHECK(ctx);
  {
    TimedLaunch tl_(ctx, KK_FLOW_FINISH);
    SCHED_CUDA_CHECK(ctx, launch_beside(ctx, flow_finish_kernel, std::min((c.num_jobs + 7) / 8, ctx->num_sms), 256, a));
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
