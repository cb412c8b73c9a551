// Host-side helpers (declared in host_util.cuh): host-thread loops, the
// stable radix order used by the planners, argument checks, and the device
// gather of saturated pairs for the exact int32 rerun (scores stay
// exact, Sec. II.B.1).
#include "host_util.cuh"

#include <algorithm>
#include <numeric>

namespace dsa {

// Host threads for a loop of n items, at least `per` items each (1 .. 16).
unsigned host_threads(size_t n, size_t per) {
  const unsigned hw = std::max(1u, std::min(16u, std::thread::hardware_concurrency()));
  return (unsigned)std::max<size_t>(1, std::min<size_t>(hw, n / std::max<size_t>(per, 1)));
}

// Stable ascending order of 64-bit keys: identity when they already are in
// order, else an LSD radix sort on 11-bit digits (digits shared by every key
// are skipped); each pass counts per host thread, then scatters in parallel
// (thread t's items of a digit follow those of threads < t: stable).
std::vector<uint32_t> radix_order(const std::vector<uint64_t>& key) {
  const size_t n = key.size();
  std::vector<uint32_t> idx(n);
  std::iota(idx.begin(), idx.end(), 0u);
  if (std::is_sorted(key.begin(), key.end())) return idx;
  uint64_t all_or = 0, all_and = ~0ull;
  for (uint64_t k : key) { all_or |= k; all_and &= k; }
  const uint64_t varying = all_or ^ all_and;
  const unsigned T = host_threads(n, 1u << 16);
  constexpr size_t B = 2048;
  std::vector<uint32_t> tmp(n);
  std::vector<uint64_t> cur(n), nxt(n);   // keys in the current order
  for (size_t x = 0; x < n; ++x) cur[x] = key[x];
  std::vector<size_t> cnt((size_t)T * B);
  for (int shift = 0; shift < 64; shift += 11) {
    if (((varying >> shift) & 0x7FFull) == 0) continue;
    std::fill(cnt.begin(), cnt.end(), 0);
    parallel_for(n, T, [&](unsigned t, size_t b, size_t e) {
      size_t* c = cnt.data() + (size_t)t * B;
      for (size_t x = b; x < e; ++x) ++c[(cur[x] >> shift) & 0x7FF];
    });
    size_t run = 0;   // exclusive offsets in (digit, thread) order
    for (size_t d = 0; d < B; ++d)
      for (unsigned t = 0; t < T; ++t) {
        const size_t c = cnt[(size_t)t * B + d];
        cnt[(size_t)t * B + d] = run;
        run += c;
      }
    parallel_for(n, T, [&](unsigned t, size_t b, size_t e) {
      size_t* c = cnt.data() + (size_t)t * B;
      for (size_t x = b; x < e; ++x) {
        const size_t dst = c[(cur[x] >> shift) & 0x7FF]++;
        tmp[dst] = idx[x];
        nxt[dst] = cur[x];
      }
    });
    idx.swap(tmp);
    cur.swap(nxt);
  }
  return idx;
}

int set_device(dsa_ctx* ctx) {
  DSA_CUDA_TRY(cudaSetDevice(ctx->device));
  return DSA_OK;
}

uint64_t memory_room(dsa_ctx* ctx) {
  if (ctx->budget) {
    std::lock_guard<std::mutex> lk(ctx->mu);
    return ctx->budget > ctx->in_use ? ctx->budget - ctx->in_use : 0;
  }
  size_t free = 0, total = 0;
  uint64_t held = 0, used = 0;
  if (cudaMemGetInfo(&free, &total) != cudaSuccess ||
      cudaMemPoolGetAttribute(ctx->pool, cudaMemPoolAttrReservedMemCurrent, &held) != cudaSuccess ||
      cudaMemPoolGetAttribute(ctx->pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess)
    cudaGetLastError();
  return free + (held > used ? held - used : 0);
}

int check_matrix(const int8_t* matrix, int A, int o, int e, Validated* v) {
  if (!matrix) { set_error("matrix is NULL"); return DSA_ERR_INVALID_ARG; }
  if (o < 0 || e < 0 || e > o) {
    set_error("gap penalties must satisfy 0 <= gap_extend <= gap_open (got %d, %d)", o, e);
    return DSA_ERR_INVALID_ARG;
  }
  int smax = -128, smin = 127;
  for (int k = 0; k < A * A; ++k) {
    smax = std::max<int>(smax, matrix[k]);
    smin = std::min<int>(smin, matrix[k]);
  }
  v->smax = smax;
  v->smin = smin;
  return DSA_OK;
}

// Band items (pair, band) of a band-pipelined score pass, in latest-start
// order.  Band b of a pair trails its predecessor, so it can start about
// b * LAG steps after the pair's first band, and the pair needs about
// n + bands * LAG steps in all; sorting the items by b * LAG - (n + bands *
// LAG) starts the longest chains first without parking warps on bands that
// are far behind their predecessors.  Inside a pair the key grows with b, so
// a band's predecessor is always taken earlier (the bounded waits rely on
// that: a warp waits only on a band some running warp holds).
std::vector<uint32_t> band_items(const std::vector<std::pair<uint32_t, uint32_t>>& mn, int band) {
  constexpr int64_t LAG = 128;
  struct It { int64_t key; uint32_t p, b; };
  std::vector<It> its;
  for (uint32_t p = 0; p < mn.size(); ++p) {
    const uint32_t nb = (mn[p].first + band - 1) / band;
    const int64_t cp = (int64_t)mn[p].second + (int64_t)nb * LAG;
    for (uint32_t b = 0; b < nb; ++b) its.push_back({(int64_t)b * LAG - cp, p, b});
  }
  std::stable_sort(its.begin(), its.end(), [](const It& x, const It& y) { return x.key < y.key; });
  std::vector<uint32_t> items;
  items.reserve(2 * its.size());
  for (const It& it : its) { items.push_back(it.p); items.push_back(it.b); }
  return items;
}

// Every S + o of the matrix fits int8 (the byte-permute substitution tables).
bool s_plus_o_fits_int8(const int8_t* matrix, int A, int o) {
  for (int x = 0; x < A * A; ++x)
    if (matrix[x] + o < -128 || matrix[x] + o > 127) return false;
  return true;
}

// Position-specific profile: the value range of its `n` entries.
int check_pssm(const int8_t* pssm, uint64_t n, int o, int e, Validated* v) {
  if (!pssm) { set_error("pssm is NULL"); return DSA_ERR_INVALID_ARG; }
  if (o < 0 || e < 0 || e > o) {
    set_error("gap penalties must satisfy 0 <= gap_extend <= gap_open (got %d, %d)", o, e);
    return DSA_ERR_INVALID_ARG;
  }
  int smax = -128, smin = 127;
  for (uint64_t k = 0; k < n; ++k) {
    smax = std::max<int>(smax, pssm[k]);
    smin = std::min<int>(smin, pssm[k]);
  }
  v->smax = smax;
  v->smin = smin;
  return DSA_OK;
}

namespace {

// Pairs whose packed pass saturated: indices gathered on the device.
__global__ void k_collect_flags(const uint8_t* __restrict__ flag, uint64_t n,
                                uint32_t* __restrict__ list, uint32_t cap,
                                uint32_t* __restrict__ count) {
  for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n;
       x += (uint64_t)gridDim.x * blockDim.x) {
    if (flag[x]) {
      const uint32_t k = atomicAdd(count, 1u);
      if (k < cap) list[k] = (uint32_t)x;
    }
  }
}

}  // namespace

int launch_collect_flags(dsa_ctx* ctx, const uint8_t* flag, uint64_t n, uint32_t* list,
                         uint32_t cap, uint32_t* count) {
  const uint64_t blk = std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->sm_count * 16);
  if (blk == 0) return DSA_OK;
  k_collect_flags<<<(unsigned)blk, 256, 0, ctx->stream>>>(flag, n, list, cap, count);
  DSA_CUDA_TRY(cudaGetLastError());
  ++ctx->launches;
  return DSA_OK;
}

}  // namespace dsa
