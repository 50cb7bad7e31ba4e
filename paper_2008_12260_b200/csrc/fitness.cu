// Population fitness (Eq. 14): per (candidate, job) row summary (K = SUM(a), N = occupied
// nodes, "row differs from the current allocation"), speedup gather, re-allocation
// penalty, floor, and the power-mean reduction over the active jobs.
//
// Two kernels stream the dense int16 population once with wide loads.
//  * fitness_kernel: rows of whole 16-byte vectors, no penalty.  Rows are split over LPR lanes (a power of
//    two <= 32); a warp summarises 32 rows, parks each row's packed (K, N) in one lane, and then
//    all 32 lanes do the gather / power term for their row at once.
//  * fitness_flat_kernel: everything else - rows of any width and alignment, the penalty, racks.  A block's
//    rows are one flat run of aligned vectors, and only those that hold something are looked at.
// A block covers a contiguous chunk of one candidate's rows; chunk sums go to a scratch array and the last
// block to arrive adds them in index order, so results are bitwise reproducible.
#include "common.cuh"
#include "fitness_common.cuh"

namespace {

__device__ __forceinline__ uint4 stream_load(const void *p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// per 32-bit word (two int16 entries): signed sum, and count of entries > 0
__device__ __forceinline__ void summarise_word(uint32_t w, int &ksum, uint32_t &npos) {
  ksum = __dp2a_lo((int)w, 0x0101, ksum);
  npos += __vimin_s16x2_relu(w, 0x00010001u);   // min(v, 1) floored at 0, per half
}

struct FitnessArgs {
  const int16_t *pop;
  const int16_t *cur;
  const float *table;
  const float *pen;       // [J] factor applied to changed rows, or NULL
  const int32_t *cur_nz;  // [J] entries of the current allocation's row that are not 0 (with pen)
  const uint8_t *active;  // or NULL
  const uint32_t *summ;   // [count][J] row summaries from the row/column kernels (SUMMARY mode)
  const float *table_rack;   // with rack: table of rows whose nodes lie in two racks or more
  const int16_t *rack;    // [num_nodes] or NULL
  int J, num_nodes, k_max, n_max;
  int lpr_log2;           // lanes per row = 1 << lpr_log2
  int rows_per_block, chunks;
  int mode;
  float p, floor_;
  double *partial;        // [count][chunks][2]: sum of terms, number of active rows
  unsigned int *ticket;   // [count]
  float *fitness;
};

// End of a block's work: its terms are added in a fixed order, the chunk sum goes to scratch,
// and the last block of the candidate to arrive adds the chunk sums in index order and
// writes the power mean.
__device__ __forceinline__ void block_finish(const FitnessArgs &a, int cand, int chunk, int j0, int j1,
                                             const float *s_term) {
  __syncthreads();
  double t, n;
  block_term_sum(s_term, j1 - j0, j0, a.active, t, n);
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    double *dst = a.partial + ((size_t)cand * a.chunks + chunk) * 2;
    dst[0] = t;
    dst[1] = n;
    __threadfence();
    const unsigned prev = atomicAdd(a.ticket + cand, 1u);
    s_last = (prev == (unsigned)a.chunks - 1u);
  }
  __syncthreads();
  if (s_last && threadIdx.x == 0) {
    __threadfence();
    const volatile double *src = a.partial + (size_t)cand * a.chunks * 2;
    double ts = 0.0, ns = 0.0;
    for (int c = 0; c < a.chunks; ++c) { ts += src[2 * c]; ns += src[2 * c + 1]; }
    a.fitness[cand] = fitness_finalise(a.mode, a.p, ts, ns);
    a.ticket[cand] = 0u;   // ready for the next call on this stream
  }
}

__global__ void __launch_bounds__(256) fitness_kernel(FitnessArgs a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int cand = blockIdx.y, chunk = blockIdx.x;
  const int LPR = 1 << a.lpr_log2, RPW = 32 >> a.lpr_log2;
  const int group = lane >> a.lpr_log2, sub = lane & (LPR - 1);
  const int row_vecs = a.num_nodes / 8;
  const int j0 = chunk * a.rows_per_block;
  const int j1 = min(a.J, j0 + a.rows_per_block);
  const char *cand_base = (const char *)(a.pop + (size_t)cand * a.J * a.num_nodes);
  const size_t row_bytes = (size_t)a.num_nodes * 2;

  __shared__ float s_term[FITNESS_MAX_ROWS_PER_BLOCK];
  TermParams tp;
  tp.table = a.table; tp.pen = nullptr; tp.active = a.active;
  tp.k_max = a.k_max; tp.n_max = a.n_max; tp.mode = a.mode; tp.p = a.p; tp.floor_ = a.floor_;
  uint32_t mine = 0;
  int myrow = -1;
  int it = 0;
  const int slots_per_fill = LPR;        // iterations that fill all 32 lanes

  // warp-uniform loop: every lane takes part in the shuffles of every iteration
  for (int jb = j0 + warp * RPW; jb < j1; jb += nwarps * RPW, ++it) {
    const int j = jb + group;
    const bool live = j < j1;
    int ksum = 0;
    uint32_t npos = 0;
    if (live) {
      const char *row = cand_base + (size_t)j * row_bytes;
      // batches of vectors per lane: all loads of a batch are issued before any is used
      constexpr int B = 8;
      for (int v0 = sub; v0 < row_vecs; v0 += LPR * B) {
        uint4 x[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
          const int v = v0 + k * LPR;
          x[k] = make_uint4(0u, 0u, 0u, 0u);
          if (v < row_vecs) x[k] = stream_load(row + (size_t)v * 16);
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
          if ((x[k].x | x[k].y | x[k].z | x[k].w) != 0u) {
            summarise_word(x[k].x, ksum, npos);
            summarise_word(x[k].y, ksum, npos);
            summarise_word(x[k].z, ksum, npos);
            summarise_word(x[k].w, ksum, npos);
          }
        }
      }
    }
    // saturate the lane-local counts so that the packed fields cannot overflow when
    // 32 lanes are added: K in bits 0..15 (<= 32 * 2047), N in bits 16..31
    int nl = (int)((npos & 0xFFFFu) + (npos >> 16));
    ksum = max(0, min(ksum, 2047));
    nl = min(nl, 2047);
    uint32_t packed = (uint32_t)ksum | ((uint32_t)nl << 16);
    for (int off = LPR >> 1; off >= 1; off >>= 1) packed += __shfl_xor_sync(0xffffffffu, packed, off);
    // lane `sub` of each group parks the row its group summarised in iteration `sub`
    if (live && sub == (it & (LPR - 1))) {
      mine = packed;
      myrow = j;
    }
    const bool flush = ((it + 1) % slots_per_fill == 0) || (jb + nwarps * RPW >= j1);
    if (flush) {
      if (myrow >= 0 && (!a.active || a.active[myrow]))
        s_term[myrow - j0] = fitness_term(tp, myrow, (int)(mine & 0xFFFFu), (int)(mine >> 16), false);
      myrow = -1;
    }
  }

  block_finish(a, cand, chunk, j0, j1, s_term);
}

// Rows of any width and alignment, with the re-allocation penalty and racks.
//
// Almost every entry of a population is zero, so a block's rows are read as one flat run of aligned
// 16-byte vectors, whatever the rows' width, and only vectors that hold something are looked at: they are
// compacted into a per-warp queue (ballot + popc) and their entries added to their rows' sums in shared
// memory.  The current allocation is read at the candidate's own entries only: a row equals it when those
// agree and it has no more entries than they (cur_nz).  Same chunks and fixed-order sums as above.
// Candidates are taken last to first: what a column repair has just written last is still in L2.
// Bound: a block's loads wait for its looking, so how many blocks an SM holds and how full the last wave is;
// 3.9 TB/s.  Measured for 300 candidates of 777 x 251 with the penalty: 31 us (98 us with loads of one
// entry); for 512 of 1024 x 256: 58 us (60 us).
constexpr int FLAT_QUEUE = 64;
__host__ __device__ constexpr int flat_blocks_per_sm(int batch) { return batch == 8 ? 4 : 5; }

__host__ __device__ inline size_t flat_smem_bytes(int rows, bool racks) { return (size_t)rows * (racks ? 16 : 8); }

template <bool RACKS, int B>
__global__ void __launch_bounds__(256, flat_blocks_per_sm(B)) fitness_flat_kernel(FitnessArgs a) {
  extern __shared__ float flat_smem[];
  __shared__ __align__(16) uint4 s_qvec[8][FLAT_QUEUE];
  __shared__ int s_qat[8][FLAT_QUEUE];
  const int rows_max = a.rows_per_block;
  float *s_term = flat_smem;                             // at the end, over the row's GPUs
  int *s_k = (int *)flat_smem;
  uint32_t *s_n = (uint32_t *)(s_k + rows_max);          // entries above 0 | entries not 0 << 14 | one differs << 31
  int *s_lo = (int *)(s_n + rows_max), *s_hi = s_lo + rows_max;   // (RACKS) lowest and highest rack
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cand = gridDim.y - 1 - blockIdx.y, chunk = blockIdx.x, NN = a.num_nodes;
  const int j0 = chunk * a.rows_per_block;
  const int j1 = min(a.J, j0 + a.rows_per_block), rows = j1 - j0;
  for (int r = tid; r < rows; r += 256) {
    s_k[r] = 0;
    s_n[r] = 0u;
    if (RACKS) { s_lo[r] = 0x7fffffff; s_hi[r] = -1; }
  }
  __syncthreads();
  const int16_t *first = a.pop + ((size_t)cand * a.J + j0) * NN;
  const int16_t *cur = a.cur ? a.cur + (size_t)j0 * NN : nullptr;
  const int entries = rows * NN;                         // at most 2048 x 8192
  const int skew = (int)(((uintptr_t)first & 15) >> 1);  // vector i holds entries 8 i - skew ..
  const int vecs = (entries + skew + 7) / 8;
  const uint4 *base = (const uint4 *)(first - skew);

  uint4 *qvec = s_qvec[warp];
  int *qat = s_qat[warp];
  int queued = 0;
  auto look = [&](int count) {       // the first `count` queued vectors, one per lane
    __syncwarp();
    if (lane < count) {
      const uint4 x = qvec[lane];
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
      const int e = 8 * qat[lane] - skew;
      int row = e < 0 ? 0 : e / NN, n = e - row * NN;
      unsigned set = 0u, other = 0u;   // bit h: entry h is not 0; it is not the current allocation's
      int c[8];
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const int v = (int)(int16_t)(w[h >> 1] >> (16 * (h & 1)));
        set |= (v != 0 ? 1u : 0u) << h;
        c[h] = v;
        if (v != 0 && cur) c[h] = (int)__ldg(cur + e + h);
      }
#pragma unroll
      for (int h = 0; h < 8; ++h) other |= (c[h] != (int)(int16_t)(w[h >> 1] >> (16 * (h & 1))) ? 1u : 0u) << h;
      // the vector's part in each of its rows
      for (int h0 = 0; h0 < 8 && (set >> h0);) {
        const int h1 = min(8, NN - n);
        const unsigned part = ((1u << h1) - 1u) & ~((1u << h0) - 1u);
        if (set & part) {
          int k = 0;
          uint32_t npos = 0u;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const unsigned m = part >> (2 * q);
            summarise_word(w[q] & ((m & 1u ? 0xFFFFu : 0u) | (m & 2u ? 0xFFFF0000u : 0u)), k, npos);
          }
          atomicAdd(&s_k[row], k);
          atomicAdd(&s_n[row], (npos & 0xFFFFu) + (npos >> 16) + ((uint32_t)__popc(set & part) << 14));
          if (other & part) atomicOr(&s_n[row], 1u << 31);
          if (RACKS) {
            int lo = 0x7fffffff, hi = -1;
#pragma unroll
            for (int h = 0; h < 8; ++h)
              if (((set & part) >> h & 1u) && (int)(int16_t)(w[h >> 1] >> (16 * (h & 1))) > 0) {
                const int r = (int)__ldg(a.rack + n + h);
                lo = min(lo, r);
                hi = max(hi, r);
              }
            atomicMin(&s_lo[row], lo);
            atomicMax(&s_hi[row], hi);
          }
        }
        ++row;
        n -= NN;                     // of entry 0, by the next row
        h0 = h1;
      }
    }
    __syncwarp();
  };
  for (int v0 = 0; v0 < vecs; v0 += 256 * B) {
    uint4 x[B];
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const int i = v0 + q * 256 + tid, e = 8 * i - skew;
      x[q] = make_uint4(0u, 0u, 0u, 0u);
      if (e >= 0 && e + 8 <= entries) {
        x[q] = stream_load(base + i);
      } else if (i < vecs) {          // the run's ragged ends
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int h = 0; h < 8; ++h)
          if (e + h >= 0 && e + h < entries) w[h >> 1] |= (uint32_t)(uint16_t)first[e + h] << (16 * (h & 1));
        x[q] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const bool nz = (x[q].x | x[q].y | x[q].z | x[q].w) != 0u;
      const unsigned bal = __ballot_sync(0xffffffffu, nz);
      if (nz) {
        const int pos = queued + __popc(bal & ((1u << lane) - 1u));
        qvec[pos] = x[q];
        qat[pos] = v0 + q * 256 + tid;
      }
      queued += __popc(bal);
      if (queued >= 32) {
        look(32);
        queued -= 32;
        if (lane < queued) {          // what is left moves to the front
          const uint4 y = qvec[32 + lane];
          const int at = qat[32 + lane];
          qvec[lane] = y;
          qat[lane] = at;
        }
        __syncwarp();
      }
    }
  }
  look(queued);
  // penalty factors and counts of the current allocation come from the kernel before this one
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
  TermParams tp;
  tp.table = a.table; tp.pen = a.pen; tp.active = a.active;
  tp.k_max = a.k_max; tp.n_max = a.n_max; tp.mode = a.mode; tp.p = a.p; tp.floor_ = a.floor_;
  for (int r = tid; r < rows; r += 256) {
    const int j = j0 + r;
    if (a.active && !a.active[j]) continue;
    const uint32_t c = s_n[r];
    const int K = max(0, s_k[r]), N = (int)(c & 0x3FFFu);
    const bool changed = a.cur && ((c >> 31) || (int)((c >> 14) & 0x3FFFu) != __ldcg(a.cur_nz + j));
    const float *table = RACKS && N >= 1 && s_lo[r] != s_hi[r] ? a.table_rack : a.table;
    const float x = __ldg(table + fitness_table_index(tp, j, K, N));
    s_term[r] = fitness_term_with(tp, x, tp.pen && changed ? __ldcg(tp.pen + j) : 1.f, changed);
  }
  block_finish(a, cand, chunk, j0, j1, s_term);
}

// Fitness from the row summaries the row / column kernels keep (K | N << 11 | entries
// differing from the current allocation << 22): no pass over the matrices.  Same chunks, same
// terms and the same fixed-order sums as fitness_kernel, hence identical bits.
__global__ void __launch_bounds__(256) fitness_summary_kernel(FitnessArgs a) {
  __shared__ float s_term[FITNESS_MAX_ROWS_PER_BLOCK];
  const int cand = blockIdx.y, chunk = blockIdx.x;
  const int j0 = chunk * a.rows_per_block;
  const int j1 = min(a.J, j0 + a.rows_per_block);
  TermParams tp;
  tp.table = a.table; tp.pen = a.pen; tp.active = a.active;
  tp.k_max = a.k_max; tp.n_max = a.n_max; tp.mode = a.mode; tp.p = a.p; tp.floor_ = a.floor_;
  for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    if (!a.active || a.active[j]) {
      const uint32_t w = a.summ[(size_t)cand * a.J + j];
      s_term[j - j0] = fitness_term(tp, j, (int)(w & 0x7FFu), (int)((w >> 11) & 0x7FFu), (w >> 22) != 0u);
    }
  }
  block_finish(a, cand, chunk, j0, j1, s_term);
}

// Effective penalty per job: the re-allocation factor when the job currently holds GPUs,
// else 1 (pending jobs are never penalised); and how many entries of its current row are not 0.
// One warp per job.  The fitness kernel behind it streams the population meanwhile.
__global__ void __launch_bounds__(256) penalty_prep_kernel(const int16_t *__restrict__ cur, const float *__restrict__ rf,
                                                           int J, int num_nodes, float *__restrict__ pen,
                                                           int32_t *__restrict__ cur_nz) {
  asm volatile("griddepcontrol.launch_dependents;");
  const int lane = threadIdx.x & 31;
  const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (j >= J) return;
  long long k = 0;
  int nz = 0;
  for (int n = lane; n < num_nodes; n += 32) {
    const int v = cur[(size_t)j * num_nodes + n];
    k += v;
    nz += v != 0;
  }
  for (int off = 16; off >= 1; off >>= 1) k += __shfl_xor_sync(0xffffffffu, k, off);
  nz = __reduce_add_sync(0xffffffffu, nz);
  if (lane == 0) {
    pen[j] = (k > 0) ? rf[j] : 1.f;
    cur_nz[j] = nz;
  }
}

// Launch geometry shared by the entry points: lanes per row so that a lane owns about four vectors
// (several loads in flight, few shuffle steps; fitness_kernel only); rows per block of about 1 MB of population, shrunk
// while the grid would leave SMs idle.
void fitness_geometry(size_t row_bytes, int J, int count, int num_sms, int &lpr_log2, int &rows_per_block, int &chunks) {
  const int row_vecs = (int)(row_bytes / 16);
  lpr_log2 = 0;
  while ((4 << lpr_log2) < row_vecs && lpr_log2 < 5) ++lpr_log2;
  rows_per_block = (int)((1u << 20) / row_bytes);
  if (rows_per_block < 256) rows_per_block = 256;
  if (rows_per_block > FITNESS_MAX_ROWS_PER_BLOCK) rows_per_block = FITNESS_MAX_ROWS_PER_BLOCK;
  if (rows_per_block > J) rows_per_block = J > 0 ? J : 1;
  while (rows_per_block > 256 &&
         (long long)count * ((J + rows_per_block - 1) / rows_per_block) < 4LL * num_sms)
    rows_per_block = (rows_per_block + 1) / 2;
  chunks = J > 0 ? (J + rows_per_block - 1) / rows_per_block : 1;
}

// The kernel for the arguments: whole aligned vectors and nothing to compare with go to fitness_kernel
// (which sums a row's vectors where they are), everything else to the flat one (which first finds the
// vectors that hold something).  after_prep: launched behind penalty_prep_kernel, so that it may start
// while that still runs.
cudaError_t launch_fitness_kernel(const FitnessArgs &a, int count, int num_sms, bool after_prep, cudaStream_t stream) {
  const dim3 grid((unsigned)a.chunks, (unsigned)count);
  const size_t row_bytes = (size_t)a.num_nodes * 2;
  if (a.summ) {
    fitness_summary_kernel<<<grid, 256, 0, stream>>>(a);
    return cudaGetLastError();
  }
  if (!a.cur && !a.rack && row_bytes % 16 == 0 && (uintptr_t)a.pop % 16 == 0) {
    fitness_kernel<<<grid, 256, 0, stream>>>(a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(256);
  lc.dynamicSmemBytes = flat_smem_bytes(a.rows_per_block, a.rack != nullptr);
  lc.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = after_prep ? 1 : 0;
  // Eight vectors per thread at once, or four and a fifth block per SM where that makes the grid a wave shorter
  const long long blocks = (long long)a.chunks * count;
  auto waves = [&](int batch) {
    const long long resident = (long long)flat_blocks_per_sm(batch) * num_sms;
    return (blocks + resident - 1) / resident;
  };
  const bool wide = waves(8) <= waves(4);
  void (*const kernel)(FitnessArgs) = a.rack ? (wide ? fitness_flat_kernel<true, 8> : fitness_flat_kernel<true, 4>)
                                             : (wide ? fitness_flat_kernel<false, 8> : fitness_flat_kernel<false, 4>);
  return cudaLaunchKernelEx(&lc, kernel, a);
}

}  // namespace

// Rows per block and blocks per candidate that launch_fitness uses for `count` candidates.
void fitness_chunking(const sched_ctx *ctx, int32_t count, int &rows_per_block, int &chunks) {
  int lpr_log2;
  fitness_geometry((size_t)ctx->cfg.num_nodes * 2, ctx->cfg.num_jobs, count, ctx->num_sms, lpr_log2, rows_per_block, chunks);
}

int launch_penalty_prep(sched_ctx *ctx, const int16_t *d_cur, const float *d_rf) {
  const int J = ctx->cfg.num_jobs;
  if (J == 0) return SCHED_OK;
  {
    TimedLaunch tl_(ctx, KK_PENPREP);
    penalty_prep_kernel<<<(J * 32 + 255) / 256, 256, 0, ctx->stream>>>(d_cur, d_rf, J, ctx->cfg.num_nodes, ctx->d_pen,
                                                                       ctx->d_cur_nz);
  }
  SCHED_LAUNCH_CHECK(ctx);
  return SCHED_OK;
}

// d_speedup_rack: table of rows whose occupied nodes lie in two or more racks, or NULL (one rack)
int launch_fitness(sched_ctx *ctx, const int16_t *d_pop, int32_t count, const float *d_speedup,
                   const int16_t *d_cur, const float *d_rf, const uint8_t *d_active, float p,
                   float *d_fitness, const uint32_t *d_summ, const float *d_speedup_rack) {
  const sched_config &c = ctx->cfg;
  const int J = c.num_jobs;
  if (count == 0) return SCHED_OK;
  if (J == 0) {     // the mean over no jobs: 0 by definition
    SCHED_CUDA_CHECK(ctx, cudaMemsetAsync(d_fitness, 0, (size_t)count * sizeof(float), ctx->stream));
    return SCHED_OK;
  }
  int lpr_log2, rows_per_block, chunks;
  fitness_geometry((size_t)c.num_nodes * 2, J, count, ctx->num_sms, lpr_log2, rows_per_block, chunks);
  int rc = ensure_fitness_scratch(ctx, count, chunks);
  if (rc != SCHED_OK) return rc;
  const bool penalise = d_cur && d_rf, prep = penalise && !ctx->pen_ready;
  if (prep && (rc = launch_penalty_prep(ctx, d_cur, d_rf)) != SCHED_OK) return rc;

  FitnessArgs a = {};
  a.cur = penalise ? d_cur : nullptr;
  a.table = d_speedup;
  a.table_rack = d_speedup_rack; a.rack = d_speedup_rack ? ctx->d_rack : nullptr;
  a.pen = penalise ? ctx->d_pen : nullptr;
  a.cur_nz = ctx->d_cur_nz;
  a.active = d_active;
  a.J = J; a.num_nodes = c.num_nodes; a.k_max = c.k_max; a.n_max = c.n_max;
  a.lpr_log2 = lpr_log2;
  a.rows_per_block = rows_per_block; a.chunks = chunks;
  a.p = p; a.floor_ = c.speedup_floor;
  a.mode = fitness_mode(p);
  // grid.y is limited to 65535 candidates per launch
  for (int32_t first = 0; first < count; first += 65535) {
    const int32_t n = (count - first < 65535) ? (count - first) : 65535;
    a.pop = d_pop + (size_t)first * J * c.num_nodes;
    a.summ = d_summ ? d_summ + (size_t)first * J : nullptr;
    a.partial = ctx->d_partial + (size_t)first * chunks * 2;
    a.ticket = ctx->d_ticket + first;
    a.fitness = d_fitness + first;
    {
      TimedLaunch tl_(ctx, KK_FITNESS);
      SCHED_CUDA_CHECK(ctx, launch_fitness_kernel(a, n, ctx->num_sms, prep && first == 0, ctx->stream));
    }
    SCHED_LAUNCH_CHECK(ctx);
  }
  return SCHED_OK;
}

// ---------------------------------------------------------------------------------------
// Fitness without any allocation: same kernels, scratch in a fixed file-scope device array.
// ---------------------------------------------------------------------------------------
#include <mutex>

namespace {

constexpr int NOALLOC_MAX_COUNT = SCHED_NOALLOC_MAX_COUNT;
constexpr int NOALLOC_MAX_JOBS = SCHED_NOALLOC_MAX_JOBS;
// Chunk sums are stored flat, candidate-major: (candidate * chunks + chunk) * 2.  The geometry
// gives at most NOALLOC_MAX_JOBS / 256 chunks per candidate unless it halves the rows of a block
// to fill the GPU, which it only does while count * chunks < 4 * SMs: a halving at most doubles
// the chunks, so count * chunks then stays below 8 * SMs.  Either way count * chunks fits
// NOALLOC_MAX_PARTIALS for every size within the documented limits (checked again per call).
constexpr size_t NOALLOC_MAX_PARTIALS = (size_t)NOALLOC_MAX_COUNT * (NOALLOC_MAX_JOBS / 256);

struct NoAllocScratch {
  double partial[NOALLOC_MAX_PARTIALS * 2];
  unsigned int ticket[NOALLOC_MAX_COUNT];
  float pen[NOALLOC_MAX_JOBS];
  int32_t cur_nz[NOALLOC_MAX_JOBS];
};

// Lives in every GPU that loads the library, from load to exit (about 2.2 MB).  In host code
// this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;
NoAllocScratch *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};
int g_noalloc_sms[NOALLOC_MAX_DEVICES] = {};
char g_noalloc_error[256] = "";

int noalloc_fail(int code, const char *msg, cudaError_t e = cudaSuccess) {
  if (e != cudaSuccess) snprintf(g_noalloc_error, sizeof(g_noalloc_error), "%s: %s", msg, cudaGetErrorString(e));
  else snprintf(g_noalloc_error, sizeof(g_noalloc_error), "%s", msg);
  return code;
}

}  // namespace

extern "C" {
#pragma GCC visibility push(default)

const char *eval_fitness_noalloc_last_error(void) { return g_noalloc_error; }

int eval_fitness_noalloc(const int16_t *d_pop, int32_t count, int32_t num_jobs, int32_t num_nodes,
                         int32_t k_max, int32_t n_max, const float *d_speedup, const int16_t *d_cur,
                         const float *d_realloc_factor, const uint8_t *d_active, float p,
                         float speedup_floor, float *d_fitness, void *cuda_stream) {
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (count < 0 || num_jobs < 1 || num_nodes < 1 || k_max < 1 || n_max < 1)
    return noalloc_fail(SCHED_ERR_INVALID_ARG, "eval_fitness_noalloc: sizes must be positive");
  if (count == 0) return SCHED_OK;
  if (!d_pop || !d_speedup || !d_fitness)
    return noalloc_fail(SCHED_ERR_INVALID_ARG, "eval_fitness_noalloc: d_pop, d_speedup and d_fitness must be non-NULL");
  if (count > NOALLOC_MAX_COUNT || num_jobs > NOALLOC_MAX_JOBS || num_nodes > SCHED_MAX_NODES ||
      k_max > SCHED_MAX_K || n_max > SCHED_MAX_N)
    return noalloc_fail(SCHED_ERR_TOO_LARGE,
                        "eval_fitness_noalloc: count <= 2048, num_jobs <= 16384, num_nodes <= 8192, "
                        "k_max, n_max <= 1024 (the scratch array is fixed; use eval_fitness beyond that)");
  if (!(p == p) || !(speedup_floor >= 0.f))
    return noalloc_fail(SCHED_ERR_INVALID_ARG, "eval_fitness_noalloc: p is NaN or speedup_floor negative");
  if (((uintptr_t)d_pop & 1) || ((uintptr_t)d_cur & 1) || ((uintptr_t)d_speedup & 3) || ((uintptr_t)d_fitness & 3))
    return noalloc_fail(SCHED_ERR_INVALID_ARG, "eval_fitness_noalloc: a buffer is not aligned to its element size");

  // set-up, once per device, with that device current: resolve the scratch array's address
  int device = -1;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return noalloc_fail(SCHED_ERR_CUDA, "cudaGetDevice", e);
  if (device < 0 || device >= NOALLOC_MAX_DEVICES)
    return noalloc_fail(SCHED_ERR_TOO_LARGE, "eval_fitness_noalloc: device ordinal beyond 63");
  if (!g_noalloc_ptr[device]) {
    void *ptr = nullptr;
    e = cudaGetSymbolAddress((void **)&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || !ptr) return noalloc_fail(SCHED_ERR_CUDA, "cudaGetSymbolAddress(scratch)", e);
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return noalloc_fail(SCHED_ERR_CUDA, "cudaDeviceGetAttribute", e);
    g_noalloc_sms[device] = sms;
    g_noalloc_ptr[device] = (NoAllocScratch *)ptr;
  }
  NoAllocScratch *scratch = g_noalloc_ptr[device];
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const int J = num_jobs;

  // the arrival counters must start at zero; the array keeps whatever the last call left
  e = cudaMemsetAsync(scratch->ticket, 0, sizeof(unsigned int) * (size_t)count, stream);
  if (e != cudaSuccess) return noalloc_fail(SCHED_ERR_CUDA, "cudaMemsetAsync(ticket)", e);

  const bool penalise = d_cur && d_realloc_factor;
  if (penalise) {
    penalty_prep_kernel<<<(J * 32 + 255) / 256, 256, 0, stream>>>(d_cur, d_realloc_factor, J, num_nodes,
                                                                 scratch->pen, scratch->cur_nz);
    e = cudaGetLastError();
    if (e != cudaSuccess) return noalloc_fail(SCHED_ERR_CUDA, "penalty_prep_kernel launch", e);
  }

  int lpr_log2, rows_per_block, chunks;
  fitness_geometry((size_t)num_nodes * 2, J, count, g_noalloc_sms[device], lpr_log2, rows_per_block, chunks);
  if ((size_t)count * (size_t)chunks > NOALLOC_MAX_PARTIALS)   // cannot happen within the limits above
    return noalloc_fail(SCHED_ERR_TOO_LARGE, "eval_fitness_noalloc: chunk sums exceed the scratch array");

  FitnessArgs a = {};
  a.pop = d_pop;
  a.cur = penalise ? d_cur : nullptr;
  a.table = d_speedup;
  a.pen = penalise ? scratch->pen : nullptr;
  a.active = d_active;
  a.cur_nz = scratch->cur_nz;
  a.J = J; a.num_nodes = num_nodes; a.k_max = k_max; a.n_max = n_max;
  a.lpr_log2 = lpr_log2;
  a.rows_per_block = rows_per_block; a.chunks = chunks;
  a.p = p; a.floor_ = speedup_floor;
  a.mode = fitness_mode(p);
  a.partial = scratch->partial;
  a.ticket = scratch->ticket;
  a.fitness = d_fitness;
  e = launch_fitness_kernel(a, count, g_noalloc_sms[device], penalise, stream);
  if (e != cudaSuccess) return noalloc_fail(SCHED_ERR_CUDA, "fitness_kernel launch", e);
  return SCHED_OK;
}

#pragma GCC visibility pop
}  // extern "C"
