// dsa_score_pairs_noalloc: the exact int32 score pass over explicit pairs
// (the map phase's per-pair scores, Sec. II.B.1), for callers that cannot
// allocate device memory.
//
// Who needs it: code that must not call cudaMalloc or any allocating
// routine -- for example an embedding application that hands every byte of
// device memory to its own pool and forbids other allocations, a
// latency-critical serving thread that may not block on the device
// allocator, or a caller recording work while allocation is not permitted.
// Such callers pass every input and output as device memory they already
// own; the only other memory this path touches is the fixed scratch array
// below, which is part of the loaded library image.
//
// It computes the same scores and end cells as dsa_align on explicit pairs, in
// two kernels.  The first aligns pairs on the packed wavefront form
// (pairwave.cuh), several lanes a pair; with the matrix on the device and no
// planner, each warp takes a run of pairs, orders it by query length and
// checks the scoring and every pair's range itself.  Pairs that form cannot
// hold (scores past 16 bits, matrices past its byte tables, local bests that
// may have wrapped) are marked, and the second kernel, one thread per pair in
// int32 (query strips of 8 rows in registers, target scanned column by column,
// the strip's last row handed on through a boundary row), does those.
//
// Bound by the ALU pipe.  30,011 reads of 36-301 bp in 411 bp windows,
// semi-global: 47.1 ms with one thread per pair for all, 1.2 ms now.
#include "pairwave.cuh"

#include <algorithm>
#include <mutex>

namespace dsa {
namespace {

// Fixed scratch for the boundary rows of every call: 4 Mi int2 = 32 MiB.
// It exists once per device that loads the library and lives until exit.
constexpr uint64_t NOALLOC_SCRATCH_ELEMS = 4ull << 20;
constexpr uint32_t NOALLOC_MAX_T_LEN = 32768;   // 128 concurrent pairs at this length
constexpr int NOALLOC_STRIP = 8;
constexpr int NOALLOC_THREADS = 128;
static __device__ __align__(256) int2 g_noalloc_scratch[NOALLOC_SCRATCH_ELEMS];

constexpr int32_t NA_TODO = -3;                 // q_end of a pair left to the second kernel

struct NoallocArgs {
  const uint8_t* qcodes;
  const uint64_t* qoff;
  uint32_t nq;
  const uint8_t* tcodes;
  const uint64_t* toff;
  uint32_t nt;
  const dsa_pair* pairs;
  uint64_t n_pairs;
  int mode;
  uint32_t fe;
  const int8_t* S;
  int A, o, e;
  uint32_t slice;                // columns of a boundary row
  int64_t bound;
  uint32_t* scratch;
  int G;                         // lanes per pair
  uint32_t per_warp;             // pairs a warp takes at once (at most 32)
  int32_t *o_score, *o_qend, *o_tend;
};

template <bool LOCAL, int MINB>
__global__ void __launch_bounds__(WAVE_WARPS * 32, MINB) k_noalloc_wave(const NoallocArgs N) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int s_max, s_min;
  constexpr unsigned FULL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) { s_max = -128; s_min = 127; }
  __syncthreads();
  for (int x = threadIdx.x; x < N.A * N.A; x += blockDim.x) {
    atomicMax(&s_max, (int)N.S[x]);
    atomicMin(&s_min, (int)N.S[x]);
  }
  __syncthreads();
  const int smax = s_max, smin = s_min;
  const int K = pair_wave_K(N.o, N.e, smin);
  const WaveParams W{N.A, N.o, N.e, N.mode, N.fe, K, pair_wave_bias(N.o, N.e, K)};
  const bool tables = pair_wave_tables_ok(LOCAL, N.o, N.e, smax, smin);
  uint8_t* const tab = smem;
  uint8_t* const prof = smem + pair_wave_table_bytes(N.A) + warp * pair_wave_warp_bytes(N.A, LOCAL);
  uint2* const park = reinterpret_cast<uint2*>(prof + pair_wave_park_offset(N.A));
  pair_wave_table<LOCAL ? WAVE_LOCAL : WAVE_GLOBAL>(W, tab, [&](int q, int a) { return (int)N.S[q * N.A + a]; });
  __syncthreads();
  const int G = N.G, per = 32 / G;
  const uint64_t gw = (uint64_t)blockIdx.x * WAVE_WARPS + warp;   // warp of the grid
  uint32_t* const scr = N.scratch + (gw * per + lane / G) * N.slice;
  const uint64_t step = (uint64_t)gridDim.x * WAVE_WARPS * N.per_warp;
  for (uint64_t p0 = gw * N.per_warp; p0 < N.n_pairs; p0 += step) {
    // lane x: pair p0 + x, its lengths (m = 0: none, not valid or left over)
    const uint32_t cnt = (uint32_t)min((uint64_t)N.per_warp, N.n_pairs - p0);
    int m = 0;
    if (lane < cnt) {
      const uint64_t p = p0 + lane;
      const dsa_pair pr = N.pairs[p];
      // pairs that break a rule get score INT32_MIN and ends -2
      bool ok = pr.query_id < N.nq && pr.target_id < N.nt && pr.t_len >= 1 && pr.t_len <= N.slice;
      if (ok) {
        m = (int)(N.qoff[pr.query_id + 1] - N.qoff[pr.query_id]);
        const uint64_t tl = N.toff[pr.target_id + 1] - N.toff[pr.target_id];
        // window inside the target, tested without the sum t_offset + t_len
        // (which wraps for offsets near 2^64)
        ok = m >= 1 && pr.t_offset <= tl && pr.t_len <= tl - pr.t_offset &&
             (int64_t)m + pr.t_len + 2 < N.bound;
      }
      if (!ok) {
        N.o_score[p] = INT32_MIN; N.o_qend[p] = -2; N.o_tend[p] = -2;
        m = 0;
      } else if (!tables || (!LOCAL && !pair_wave_range_ok(m, pr.t_len, N.o, N.e, smax, smin))) {
        N.o_qend[p] = NA_TODO;
        m = 0;
      }
    }
    // order by query length, longest first, so that a bundle's pairs take
    // about the same rows; pairs already decided go last
    int rank = 0;
    for (int x = 0; x < 32; ++x) {
      const int mx = __shfl_sync(FULL, m, x);
      rank += mx > m || (mx == m && x < lane);
    }
    const uint32_t live = __popc(__ballot_sync(FULL, m > 0));
    for (uint32_t at = 0; at < live; at += per) {
      // the group's pair: the lane whose rank is at + group
      const uint32_t want = at + lane / G;
      int src = -1;
      for (int x = 0; x < 32; ++x)
        if ((uint32_t)__shfl_sync(FULL, rank, x) == want) src = x;
      const bool has = want < live;
      const uint64_t p = p0 + (uint32_t)max(src, 0);
      const uint8_t *q = nullptr, *t = nullptr;
      int mm = 0, nn = 0;
      bool ok = true;
      if (has) {
        const dsa_pair pr = N.pairs[p];
        q = N.qcodes + N.qoff[pr.query_id];
        t = N.tcodes + N.toff[pr.target_id] + pr.t_offset;
        mm = (int)(N.qoff[pr.query_id + 1] - N.qoff[pr.query_id]);
        nn = (int)pr.t_len;
        // every residue code must index the matrix
        for (int x = lane & (G - 1); x < mm; x += G) ok = ok && q[x] < N.A;
        for (int x = lane & (G - 1); x < nn; x += G) ok = ok && t[x] < N.A;
      }
      for (int w = G / 2; w > 0; w >>= 1) ok = __shfl_xor_sync(FULL, ok ? 1 : 0, w) && ok;
      const bool first = has && (lane & (G - 1)) == 0;
      if (!ok) {
        if (first) { N.o_score[p] = INT32_MIN; N.o_qend[p] = -2; N.o_tend[p] = -2; }
        mm = nn = 0;
      }
      int mmax = mm;
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) mmax = max(mmax, __shfl_xor_sync(FULL, mmax, w));
      int s, i, j;
      if (mmax <= 16 * G)
        pair_wave_run<LOCAL ? WAVE_LOCAL : WAVE_GLOBAL, 8>(W, tab, prof, park, G, q, t, mm, nn, scr, s, i, j);
      else if (mmax <= 24 * G)
        pair_wave_run<LOCAL ? WAVE_LOCAL : WAVE_GLOBAL, 12>(W, tab, prof, park, G, q, t, mm, nn, scr, s, i, j);
      else
        pair_wave_run<LOCAL ? WAVE_LOCAL : WAVE_GLOBAL, 16>(W, tab, prof, park, G, q, t, mm, nn, scr, s, i, j);
      if (first && ok) {
        const bool wrapped = LOCAL && s > 32767 - max(0, smax);
        N.o_score[p] = s;
        N.o_qend[p] = wrapped ? NA_TODO : i - 1;
        N.o_tend[p] = j - 1;
      }
      __syncwarp();
    }
  }
}

__device__ __forceinline__ int32_t na_row0(int mode, uint32_t fe, int64_t j, int o, int e) {
  if (j == 0 || mode == DSA_LOCAL || (mode == DSA_SEMIGLOBAL && (fe & DSA_FREE_T_BEGIN))) return 0;
  return -(o + (int32_t)(j - 1) * e);
}
__device__ __forceinline__ int32_t na_col0(int mode, uint32_t fe, int64_t i, int o, int e) {
  if (i == 0 || mode == DSA_LOCAL || (mode == DSA_SEMIGLOBAL && (fe & DSA_FREE_Q_BEGIN))) return 0;
  return -(o + (int32_t)(i - 1) * e);
}

// The pairs that the first kernel left over.
__global__ void __launch_bounds__(NOALLOC_THREADS) k_noalloc_pairs(
    const uint8_t* __restrict__ qcodes, const uint64_t* __restrict__ qoff,
    const uint8_t* __restrict__ tcodes, const uint64_t* __restrict__ toff,
    const dsa_pair* __restrict__ pairs, uint64_t n_pairs, int mode, uint32_t fe,
    const int8_t* __restrict__ Sg, int A, int o, int e, uint32_t slice,
    int2* __restrict__ scratch, int32_t* __restrict__ o_score, int32_t* __restrict__ o_qend,
    int32_t* __restrict__ o_tend) {
  __shared__ int8_t S[32 * 32];
  for (int x = threadIdx.x; x < A * A; x += blockDim.x) S[x] = Sg[x];
  __syncthreads();
  const bool local = mode == DSA_LOCAL;
  const bool sg = mode == DSA_SEMIGLOBAL;
  const bool q_end_free = sg && (fe & DSA_FREE_Q_END);
  const bool t_end_free = sg && (fe & DSA_FREE_T_END);
  const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  int2* scr = scratch + tid * slice;   // this thread's boundary row
  for (uint64_t p = tid; p < n_pairs; p += (uint64_t)gridDim.x * blockDim.x) {
    if (o_qend[p] != NA_TODO) continue;   // done by the first kernel
    const dsa_pair pr = pairs[p];
    const int32_t m = (int32_t)(qoff[pr.query_id + 1] - qoff[pr.query_id]);
    bool ok = true;   // ids, window and lengths were checked there
    {   // every residue code must index the matrix
      const uint8_t* qq = qcodes + qoff[pr.query_id];
      const uint8_t* tt = tcodes + toff[pr.target_id] + pr.t_offset;
      for (int32_t i = 0; i < m && ok; ++i) ok = qq[i] < A;
      for (uint32_t j = 0; j < pr.t_len && ok; ++j) ok = tt[j] < A;
    }
    if (!ok) {
      o_score[p] = INT32_MIN; o_qend[p] = -2; o_tend[p] = -2;
      continue;
    }
    const int32_t n = (int32_t)pr.t_len;
    const uint8_t* q = qcodes + qoff[pr.query_id];
    const uint8_t* t = tcodes + toff[pr.target_id] + pr.t_offset;
    int32_t bs = 0, bi = -1, bj = -1;
    bool have = false;
    auto offer = [&](int32_t h, int32_t ii, int32_t jj) {
      if (!have || h > bs || (h == bs && (jj < bj || (jj == bj && ii < bi)))) {
        bs = h; bi = ii; bj = jj; have = true;
      }
    };
    if (q_end_free) offer(na_row0(mode, fe, n, o, e), 0, n);
    for (int32_t i0 = 0; i0 < m; i0 += NOALLOC_STRIP) {
      const int rows = min(NOALLOC_STRIP, m - i0);
      int32_t Hc[NOALLOC_STRIP], Ec[NOALLOC_STRIP];
      int qc[NOALLOC_STRIP];
#pragma unroll
      for (int r = 0; r < NOALLOC_STRIP; ++r) {
        Hc[r] = na_col0(mode, fe, i0 + r + 1, o, e);
        Ec[r] = NEG32;
        qc[r] = r < rows ? q[i0 + r] * A : 0;
      }
      if (t_end_free && i0 + rows == m) offer(Hc[rows - 1], m, 0);
      int32_t diag = na_col0(mode, fe, i0, o, e);
      for (int32_t j = 1; j <= n; ++j) {
        const int a = t[j - 1];
        int32_t Hup, Fup;
        if (i0 == 0) {
          Hup = na_row0(mode, fe, j, o, e);
          Fup = NEG32;
        } else {
          const int2 v = scr[j - 1];
          Hup = v.x;
          Fup = v.y;
        }
        int32_t d = diag;
        diag = Hup;
        int32_t F = Fup, Hprev = Hup;
#pragma unroll
        for (int r = 0; r < NOALLOC_STRIP; ++r) {
          if (r < rows) {
            F = max(F - e, Hprev - o);
            Ec[r] = max(Ec[r] - e, Hc[r] - o);
            int32_t h = max(d + S[qc[r] + a], max(Ec[r], F));
            if (local) h = max(h, 0);
            d = Hc[r];
            Hc[r] = h;
            Hprev = h;
            const int32_t i = i0 + r + 1;
            if (local) {
              if (h > 0) offer(h, i, j);
            } else {
              if (j == n && (q_end_free || i == m)) offer(h, i, j);
              if (t_end_free && i == m) offer(h, i, j);
            }
          }
        }
        scr[j - 1] = make_int2(Hprev, F);
      }
    }
    if (local && !have) {
      o_score[p] = 0; o_qend[p] = -1; o_tend[p] = -1;
    } else {
      o_score[p] = bs; o_qend[p] = bi - 1; o_tend[p] = bj - 1;
    }
  }
}

// Device address of g_noalloc_scratch per device, looked up once per device
// (with that device current) on the first call made on it, which also loads every
// kernel a later call may take: a kernel is otherwise loaded, into device memory,
// by the first call in its mode.  The address belongs to the device's primary
// context: it does not survive a cudaDeviceReset of that device (the header says
// so).
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[64] = {};

using WaveKernel = void (*)(const NoallocArgs);
// by mode and by whether 4 CTAs' profiles fit an SM
constexpr WaveKernel WAVE_KERNELS[2][2] = {{k_noalloc_wave<false, 2>, k_noalloc_wave<false, 4>},
                                           {k_noalloc_wave<true, 2>, k_noalloc_wave<true, 4>}};
cudaError_t load_kernels() {
  cudaFuncAttributes a;
  cudaError_t err = cudaFuncGetAttributes(&a, k_noalloc_pairs);
  for (const auto& of_mode : WAVE_KERNELS)
    for (const WaveKernel k : of_mode)
      if (err == cudaSuccess) err = cudaFuncGetAttributes(&a, k);
  return err;
}

}  // namespace
}  // namespace dsa

using namespace dsa;

extern "C" int dsa_score_pairs_noalloc(const uint8_t* d_q_codes, const uint64_t* d_q_offsets,
                                       uint32_t n_queries, const uint8_t* d_t_codes,
                                       const uint64_t* d_t_offsets, uint32_t n_targets,
                                       const dsa_pair* d_pairs, uint64_t n_pairs, int mode,
                                       uint32_t free_ends, const int8_t* d_matrix,
                                       int alphabet_size, int gap_open, int gap_extend,
                                       uint32_t max_t_len, int32_t* d_score, int32_t* d_q_end,
                                       int32_t* d_t_end, void* cuda_stream) {
  if (!d_q_codes || !d_q_offsets || !d_t_codes || !d_t_offsets || !d_pairs || !d_matrix ||
      !d_score || !d_q_end || !d_t_end) {
    set_error("dsa_score_pairs_noalloc: NULL pointer argument");
    return DSA_ERR_INVALID_ARG;
  }
  if (mode < DSA_LOCAL || mode > DSA_SEMIGLOBAL || free_ends > 15 || alphabet_size < 1 ||
      alphabet_size > MAX_ALPHABET || gap_extend < 0 || gap_extend > gap_open) {
    set_error("dsa_score_pairs_noalloc: bad mode, free_ends, alphabet_size or gap penalties");
    return DSA_ERR_INVALID_ARG;
  }
  if (max_t_len == 0 || max_t_len > NOALLOC_MAX_T_LEN) {
    set_error("dsa_score_pairs_noalloc: max_t_len %u outside 1..%u (the fixed scratch holds "
              "%llu boundary cells)", max_t_len, NOALLOC_MAX_T_LEN,
              (unsigned long long)NOALLOC_SCRATCH_ELEMS);
    return DSA_ERR_INVALID_ARG;
  }
  if (n_pairs == 0) return DSA_OK;
  int dev = 0;
  DSA_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) { set_error("device index %d unsupported", dev); return DSA_ERR_UNSUPPORTED; }
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      cudaError_t err = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (err != cudaSuccess || !p) {
        set_error("cudaGetSymbolAddress(g_noalloc_scratch) failed: %s", cudaGetErrorString(err));
        return DSA_ERR_CUDA;
      }
      DSA_CUDA_TRY(load_kernels());
      g_noalloc_ptr[dev] = p;
    }
    scratch = g_noalloc_ptr[dev];
  }
  // weight bound for int32 safety, as in dsa_align: (m + n) * max(|S|, o, e) < 2^29;
  // the matrix is on the device, so the bound uses the int8 range
  const int64_t w = std::max<int64_t>({128, gap_open, gap_extend});
  const int64_t bound = ((1ll << 29) / (w + 1));
  const uint32_t slice = max_t_len;
  const uint64_t max_threads = NOALLOC_SCRATCH_ELEMS / slice;
  uint64_t threads = std::min<uint64_t>(max_threads, n_pairs);
  uint64_t blocks = (threads + NOALLOC_THREADS - 1) / NOALLOC_THREADS;
  if (blocks * NOALLOC_THREADS > max_threads) blocks = max_threads / NOALLOC_THREADS;
  if (blocks == 0) blocks = 1;
  const cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // the wavefront kernel: as many warps as are resident at once, and as many
  // lanes a pair as it takes to keep them busy (8 when pairs abound: the fewer
  // lanes, the fewer steps a pair spends filling its wavefront)
  const bool local = mode == DSA_LOCAL;
  const size_t smem = pair_wave_smem(alphabet_size, local);
  const WaveKernel kern = WAVE_KERNELS[local][smem <= 50 * 1024];
  int sms = 0, per_sm = 0;
  DSA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DSA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)pair_wave_smem(MAX_ALPHABET, local)));
  DSA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, WAVE_WARPS * 32, smem));
  const uint64_t resident = (uint64_t)std::max(1, per_sm) * sms * WAVE_WARPS;   // warps
  NoallocArgs N{d_q_codes, d_q_offsets, n_queries, d_t_codes, d_t_offsets, n_targets, d_pairs, n_pairs,
                mode, free_ends, d_matrix, alphabet_size, gap_open, gap_extend, slice, bound,
                static_cast<uint32_t*>(scratch), 8, 0, d_score, d_q_end, d_t_end};
  while (N.G < 32 && n_pairs * N.G < resident * 32) N.G *= 2;
  const uint64_t per = 32 / N.G;
  // boundary rows bound the groups: 2 words of scratch per element
  const uint64_t scr_warps = 2 * NOALLOC_SCRATCH_ELEMS / slice / per;
  const uint64_t warps = std::max<uint64_t>(
      WAVE_WARPS, std::min({resident, scr_warps, (n_pairs + per - 1) / per}));
  const uint64_t share = (n_pairs + warps - 1) / warps;   // pairs of a warp, in whole bundles
  N.per_warp = (uint32_t)std::min<uint64_t>(32, (share + per - 1) / per * per);
  uint64_t wave_blocks = (warps + WAVE_WARPS - 1) / WAVE_WARPS;
  if (wave_blocks * WAVE_WARPS > scr_warps) wave_blocks = scr_warps / WAVE_WARPS;
  kern<<<(unsigned)wave_blocks, WAVE_WARPS * 32, smem, st>>>(N);
  DSA_CUDA_TRY(cudaGetLastError());
  k_noalloc_pairs<<<(unsigned)blocks, NOALLOC_THREADS, 0, st>>>(
      d_q_codes, d_q_offsets, d_t_codes, d_t_offsets, d_pairs, n_pairs, mode, free_ends, d_matrix,
      alphabet_size, gap_open, gap_extend, slice, static_cast<int2*>(scratch), d_score, d_q_end,
      d_t_end);
  DSA_CUDA_TRY(cudaGetLastError());
  return DSA_OK;
}
