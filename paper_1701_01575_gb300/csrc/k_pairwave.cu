// Explicit pairs as wavefronts of small lane groups (pairwave.cuh): the
// planned kernel behind dsa_align's explicit pairs (the map phase's per-pair
// scores, Sec. II.B.1, of rescoring lists and distance matrices).  The device
// planner sorts the pairs by (class, window length); a class fixes the group
// size and the rows per block, so that a query wastes at most a third of its
// rows, and the groups of a warp hold pairs of nearly equal work.  Persistent
// warps pop bundles of 32 / G pairs, the costliest class and the longest
// windows first.  Large calls of pairs that the classes mostly pad take the
// per-thread form (pairs_thread_form).
//
// Bound by the ALU pipe and, at the end of a call, by the longest pair's
// chain.  Measured against the forms it replaces (whole call): 20,000 protein
// pairs of 50-1,500 residues, local, 135 -> 2.61 ms (one thread per two
// pairs, two table loads per packed cell); 15,001 such pairs, global, 244 ->
// 1.49 ms (one thread per pair in int32, their range being past that form's
// rule); 1,000 reads of 150 bp in 500 bp windows with traceback 1.76 -> 0.64 ms; 1,000,000 of
// 150 and 250 bp, 27.4 -> 23.5 ms.
#include "pairwave.cuh"
#include "host_util.cuh"

namespace dsa {
namespace {

struct WaveRange { uint32_t first, n, item0; int G, R; };   // sorted pairs and bundles of a class
struct WaveKernelArgs {
  WaveParams W;
  const dsa_pair* pairs;
  const uint32_t* order;          // sorted pair indices
  const uint8_t* qcodes;
  const uint64_t* qoff;
  const uint32_t* qlen;
  const uint8_t* tcodes;
  const uint64_t* toff;
  const int8_t* S;
  WaveRange cls[WAVE_CLASSES];    // descending cost: cls[x] is class WAVE_CLASSES - 1 - x
  uint32_t n_items;
  uint32_t* counter;
  uint32_t* scratch;              // per warp: boundary row of multi-band pairs
  uint32_t scratch_cols;
  int T;
  Scores out;
};

template <int FORM, bool WIDE, int MINB>
__global__ void __launch_bounds__(WAVE_WARPS * 32, MINB) k_pair_wave(const WaveKernelArgs A) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr unsigned FULL = 0xFFFFFFFFu;
  constexpr bool LOCAL = FORM != WAVE_GLOBAL;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t* const tab = smem;
  uint8_t* const prof = smem + pair_wave_table_bytes(A.W.A) + warp * pair_wave_warp_bytes(A.W.A, LOCAL);
  uint2* const park = reinterpret_cast<uint2*>(prof + pair_wave_park_offset(A.W.A));
  pair_wave_table<FORM>(A.W, tab, [&](int q, int a) { return (int)A.S[q * A.W.A + a]; });
  __syncthreads();
  uint32_t* const scr = A.scratch + (uint64_t)(blockIdx.x * WAVE_WARPS + warp) * A.scratch_cols;

  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(A.counter, 1u);
    item = __shfl_sync(FULL, item, 0);
    if (item >= A.n_items) break;
    int x = 0;
    while (x + 1 < WAVE_CLASSES && item >= A.cls[x + 1].item0) ++x;
    const WaveClass C{A.cls[x].G, A.cls[x].R};
    const uint32_t per = 32u / C.G;
    const uint32_t at = (item - A.cls[x].item0) * per + lane / C.G;   // from the longest window down
    const uint8_t *q = nullptr, *t = nullptr;
    int m = 0, n = 0;
    uint32_t id = NONE;
    if (at < A.cls[x].n) {
      id = A.order[A.cls[x].first + A.cls[x].n - 1 - at];
      const dsa_pair p = A.pairs[id];
      q = A.qcodes + A.qoff[p.query_id];
      t = A.tcodes + A.toff[p.target_id] + p.t_offset;
      m = (int)A.qlen[p.query_id];
      n = (int)p.t_len;
    }
    int s, i, j;
    if (WIDE && C.R == 20)
      pair_wave_run<FORM, WIDE ? 20 : 16>(A.W, tab, prof, park, C.G, q, t, m, n, scr, s, i, j);
    else if (C.R == 16)
      pair_wave_run<FORM, 16>(A.W, tab, prof, park, C.G, q, t, m, n, scr, s, i, j);
    else if (C.R == 12)
      pair_wave_run<FORM, 12>(A.W, tab, prof, park, C.G, q, t, m, n, scr, s, i, j);
    else
      pair_wave_run<FORM, 8>(A.W, tab, prof, park, C.G, q, t, m, n, scr, s, i, j);
    if (id != NONE && (lane & (C.G - 1)) == 0) {
      A.out.score[id] = s;
      A.out.q_end[id] = i - 1;
      A.out.t_end[id] = j - 1;
      A.out.flag[id] = LOCAL && s > A.T ? 1 : 0;
    }
    __syncwarp();
  }
}

}  // namespace

static int pair_wave_group(int cls) { return wave_class(cls).G; }
bool pair_wave_wide(int A) { return A <= WAVE_WIDE_ALPHABET; }

int launch_pair_wave(dsa_ctx* ctx, const dsa_db* db, const dsa_db* qs, const int8_t* d_matrix, int A,
                     int o, int e, int mode, uint32_t fe, int smax, int smin, const dsa_pair* d_pairs,
                     const uint32_t* d_order, const uint64_t* class_n, uint32_t max_n, Scores out) {
  const bool local = mode == DSA_LOCAL;
  WaveKernelArgs K{};
  const int k = pair_wave_K(o, e, smin);
  const bool lsum = local && pair_wave_local_sum_ok(qs->max_len, max_n, o, e, smax, smin);
  K.W = {A, o, e, mode, fe, k, lsum ? 512 + o + 64 * e : pair_wave_bias(o, e, k)};
  K.pairs = d_pairs;
  K.order = d_order;
  K.qcodes = qs->d_codes; K.qoff = qs->d_off; K.qlen = qs->d_len;
  K.tcodes = db->d_codes; K.toff = db->d_off;
  K.S = d_matrix;
  uint64_t first[WAVE_CLASSES + 1] = {0};
  for (int c = 0; c < WAVE_CLASSES; ++c) first[c + 1] = first[c] + class_n[c];
  uint64_t items = 0;
  for (int x = 0; x < WAVE_CLASSES; ++x) {
    const int c = WAVE_CLASSES - 1 - x;
    const uint64_t per = 32 / pair_wave_group(c);
    K.cls[x] = {(uint32_t)first[c], (uint32_t)class_n[c], (uint32_t)items, wave_class(c).G, wave_class(c).R};
    items += (class_n[c] + per - 1) / per;
  }
  if (items == 0) return DSA_OK;
  K.n_items = (uint32_t)items;
  K.T = 32767 - std::max(0, smax);
  K.out = out;
  const size_t smem = pair_wave_smem(A, local);
  // small alphabets: registers bound the warps per SM (4 CTAs); larger ones:
  // the profiles do (2 CTAs of 4 x 28 KB for proteins)
  auto kern = pair_wave_wide(A) ? (lsum    ? k_pair_wave<WAVE_LOCAL_SUM, true, 4>
                                   : local ? k_pair_wave<WAVE_LOCAL, true, 4>
                                           : k_pair_wave<WAVE_GLOBAL, true, 4>)
                                : (lsum    ? k_pair_wave<WAVE_LOCAL_SUM, false, 2>
                                   : local ? k_pair_wave<WAVE_LOCAL, false, 2>
                                           : k_pair_wave<WAVE_GLOBAL, false, 2>);
  DSA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)pair_wave_smem(MAX_ALPHABET, local)));
  int per_sm = 0;
  DSA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, WAVE_WARPS * 32, smem));
  const uint64_t grid = std::min<uint64_t>((items + WAVE_WARPS - 1) / WAVE_WARPS,
                                           (uint64_t)std::max(1, per_sm) * ctx->sm_count);
  // only queries past one band (more than 1,024 rows) use the boundary row
  const bool multi = class_n[WAVE_CLASSES - 1] + class_n[WAVE_CLASSES - 2] != 0;
  K.scratch_cols = multi ? std::min<uint32_t>(max_n, (uint32_t)(LONG_PAIR_CELLS / 1024)) : 0;
  const size_t scr_bytes = std::max<size_t>(16, (size_t)grid * WAVE_WARPS * K.scratch_cols * 4);
  void* scr = nullptr;
  DSA_TRY(ctx->alloc(&scr, scr_bytes));
  K.scratch = static_cast<uint32_t*>(scr);
  K.counter = ctx->d_counters;
  cudaError_t err = cudaMemsetAsync(K.counter, 0, sizeof(uint32_t), ctx->stream);
  if (err == cudaSuccess) {
    kern<<<(unsigned)grid, WAVE_WARPS * 32, smem, ctx->stream>>>(K);
    ++ctx->launches;
    err = cudaGetLastError();
  }
  ctx->release(scr, scr_bytes);
  if (err != cudaSuccess) {
    set_error("k_pair_wave launch: %s", cudaGetErrorString(err));
    return DSA_ERR_CUDA;
  }
  return DSA_OK;
}

}  // namespace dsa
