// All-vs-all score pass (the map phase's per-pair scores of every query
// against every database sequence, Sec. II.B.1; DSW / DNW / DSG of
// Sec. II.C.2): the packed int16x2 path (inter-sequence kernel for most
// targets, wavefront kernel for the longest, with the autotuned split between
// them), the exact int32 rerun of saturated pairs, and the exact int32 kernel
// for searches the packed path cannot take.
#include "host_util.cuh"

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <numeric>
#include <string>
#include <sys/stat.h>
#include <unistd.h>

namespace dsa {
namespace {


// ---- autotuner: kernel variant and long-target threshold of the packed path ----
//
// Two speed choices of the packed path (every choice gives the same exact
// results): the strip height of the inter-sequence kernel (28 rows, or 20
// rows, which wastes fewer padding rows on short queries), and which
// targets go to the wavefront kernel (long) and which to the inter-sequence
// kernel.  For a workload shape (GPU, driver, kernel form, mode, alphabet,
// how far the queries fill their strips, and log2 bins of the query count, query residues, longest query, target
// count, database residues and longest target) the first call times each
// strip height at the modelled threshold (a switch needs a 2% gain), then
// every target on the wavefronts, then a local search of thresholds lower and
// higher by factors of 4 while it keeps improving by 2% or more -- and keeps
// both in a JSON cache file.  DSA_AUTOTUNE=off (28 rows, the model) | cache
// (default: tune on a miss) | retune (always tune); DSA_AUTOTUNE_CACHE names
// the file (default $XDG_CACHE_HOME/dsa/autotune.json or
// ~/.cache/dsa/autotune.json); DSA_INTER_ROWS (28 | 20) and
// DSA_LONG_THRESHOLD fix their choice.
struct Tuner {
  std::mutex mu;
  bool loaded = false;
  std::string path;
  std::map<std::string, uint32_t> cache;
};
Tuner& tuner() {
  static Tuner t;
  return t;
}

std::string tune_cache_path() {
  if (const char* p = getenv("DSA_AUTOTUNE_CACHE")) return p;
  std::string dir;
  if (const char* x = getenv("XDG_CACHE_HOME")) dir = x;
  else if (const char* h = getenv("HOME")) dir = std::string(h) + "/.cache";
  else return "";
  return dir + "/dsa/autotune.json";
}

// flat JSON object of "key": unsigned integer
void tune_load(Tuner& t, const std::string& path) {
  t.loaded = true;
  t.path = path;
  t.cache.clear();
  if (t.path.empty()) return;
  FILE* f = fopen(t.path.c_str(), "rb");
  if (!f) return;
  std::string txt;
  char buf[4096];
  size_t n;
  while ((n = fread(buf, 1, sizeof buf, f)) > 0) txt.append(buf, n);
  fclose(f);
  size_t pos = 0;
  for (;;) {
    const size_t k0 = txt.find('"', pos);
    if (k0 == std::string::npos) break;
    const size_t k1 = txt.find('"', k0 + 1);
    if (k1 == std::string::npos) break;
    const size_t c = txt.find(':', k1);
    if (c == std::string::npos) break;
    char* endp = nullptr;
    const unsigned long long val = strtoull(txt.c_str() + c + 1, &endp, 10);
    if (endp == txt.c_str() + c + 1) break;
    t.cache[txt.substr(k0 + 1, k1 - k0 - 1)] =
        (uint32_t)std::min<unsigned long long>(val, UINT32_MAX);
    pos = (size_t)(endp - txt.c_str());
  }
}

void tune_store(Tuner& t) {
  if (t.path.empty()) return;
  const size_t slash = t.path.rfind('/');
  if (slash != std::string::npos) {
    // create the directory chain (failures are ignored: the cache is optional)
    const std::string d = t.path.substr(0, slash);
    for (size_t k = 1; k <= d.size(); ++k)
      if (k == d.size() || d[k] == '/') mkdir(d.substr(0, k).c_str(), 0755);
  }
  const std::string tmp = t.path + ".tmp" + std::to_string((long long)getpid());
  FILE* f = fopen(tmp.c_str(), "wb");
  if (!f) return;
  fputs("{\n", f);
  size_t k = 0;
  for (const auto& kv : t.cache)
    fprintf(f, "  \"%s\": %u%s\n", kv.first.c_str(), kv.second, ++k < t.cache.size() ? "," : "");
  fputs("}\n", f);
  fclose(f);
  rename(tmp.c_str(), t.path.c_str());
}

int ilog2_bin(uint64_t x) {
  int b = 0;
  while (x > 1) { x >>= 1; ++b; }
  return b;
}

// Stream plan of the inter-sequence and wavefront kernels: queries, cut into
// strips of W rows, are dealt, longest first, to the currently shortest of K
// lanes (K about total / longest, so a lane is about as long as the longest
// query, or as `at_least` strips); lanes are then paired by length into units,
// low half = first lane, high half = second.  A pair of unequal lanes wastes the
// difference, so fewer lanes are taken where they waste less (5 queries of
// 60-700: 33 packed strips of 24 rows with 2 lanes, 39 with 4, the local search
// of 60,000 targets 7.2 -> 5.9 ms).  dual: both halves of a unit follow one
// lane, against two targets.
struct Streams {
  std::vector<StripMeta> meta;
  std::vector<uint32_t> sbase, ns;   // per unit: first strip, strips
};
Streams build_streams(const dsa_db* qs, const std::vector<uint32_t>& qorder, uint32_t W,
                      uint64_t at_least = 1, bool dual = false) {
  const uint32_t nq = qs->n;
  auto strips_of = [&](uint32_t q) { return (qs->h_len[q] + W - 1) / W; };
  uint64_t tot = 0, maxq = at_least;
  for (uint32_t q = 0; q < nq; ++q) {
    tot += strips_of(q);
    maxq = std::max<uint64_t>(maxq, strips_of(q));
  }
  const uint32_t most = std::min<uint32_t>((uint32_t)std::max<uint64_t>(1, (tot + maxq - 1) / maxq), nq);
  std::vector<std::vector<uint32_t>> lanes;
  std::vector<uint64_t> load;
  std::vector<uint32_t> lorder;
  auto deal = [&](uint32_t K) -> uint64_t {   // strips of all units
    lanes.assign(K, {});
    load.assign(K, 0);
    for (uint32_t q : qorder) {
      const uint32_t l = (uint32_t)(std::min_element(load.begin(), load.end()) - load.begin());
      lanes[l].push_back(q);
      load[l] += strips_of(q);
    }
    lorder.resize(K);
    std::iota(lorder.begin(), lorder.end(), 0u);
    std::stable_sort(lorder.begin(), lorder.end(), [&](uint32_t a, uint32_t b) { return load[a] > load[b]; });
    uint64_t strips = 0;
    for (uint32_t l = 0; l < K; l += dual ? 1 : 2) strips += load[lorder[l]];
    return strips;
  };
  uint32_t K = dual ? most : (most + 1) & ~1u;   // even: lanes come in pairs
  if (dual || K < 4) {
    deal(K);
  } else {
    const uint64_t more = deal(K), fewer = deal(K - 2);
    if (fewer < more) K -= 2;
    else deal(K);
  }
  Streams S;
  // query and strip index (with the LAST bit) of strip s of a lane, in order
  auto fill = [&](const std::vector<uint32_t>& lane, uint64_t n, auto put) {
    uint64_t s = 0;
    for (uint32_t x : lane) {
      const uint32_t ns_q = strips_of(x);
      for (uint32_t k = 0; k < ns_q; ++k) put(s++, x, k | (k == ns_q - 1 ? LAST : 0u));
    }
    for (; s < n; ++s) put(s, NONE, 0u);
  };
  for (uint32_t u = 0; dual && u < K; ++u) {
    const size_t at = S.meta.size();
    S.sbase.push_back((uint32_t)at);
    S.ns.push_back((uint32_t)load[u]);
    S.meta.resize(at + load[u]);
    fill(lanes[u], load[u], [&](uint64_t st, uint32_t q, uint32_t k) { S.meta[at + st] = {q, k, q, k}; });
  }
  for (uint32_t u = 0; !dual && u < K / 2; ++u) {
    const uint64_t ns_u = std::max(load[lorder[2 * u]], load[lorder[2 * u + 1]]);
    if (ns_u == 0) continue;
    const size_t at = S.meta.size();
    S.sbase.push_back((uint32_t)at);
    S.ns.push_back((uint32_t)ns_u);
    S.meta.resize(at + ns_u);
    fill(lanes[lorder[2 * u]], ns_u, [&](uint64_t st, uint32_t q, uint32_t k) { S.meta[at + st].qa = q; S.meta[at + st].ka = k; });
    fill(lanes[lorder[2 * u + 1]], ns_u, [&](uint64_t st, uint32_t q, uint32_t k) { S.meta[at + st].qb = q; S.meta[at + st].kb = k; });
  }
  return S;
}

// Cycles of the wavefronts over the first n_groups groups of the database on
// strips of R rows: the work, every unit's strips in whole bands of the lanes that
// each target takes, at 4 warps a scheduler; or the longest target's chain, its
// columns times the unit's bands, where its warp has 1.5 others beside it.  A
// warp's step takes about 11 cycles a row and 45 (global 8 and 66) for the
// hand-over.  Against the times of 134 searches of 1 to 100 queries of 32 to 2,300
// and 300 to 150,000 targets up to 100,000, the height of the smaller estimate is
// 0.3% slower than the better one on average; strips alone, without their bands,
// chose up to 53% wrong (one query of 1,000 against 4,000 targets up to 9,000, two
// bands either way: 24 rows 12.6 ms, 16 rows 8.8, the kernel before 11.2).
double wave_cycles(const dsa_ctx* ctx, const dsa_db* db, const dsa_db* qs, uint32_t n_groups,
                   uint64_t residues, uint32_t R, bool dual, bool local) {
  const uint64_t slots = 512ull * ctx->sm_count, halves = dual ? 2 : 1, longest = db->h_glen[0];
  uint64_t strips = 0;
  for (uint32_t m : qs->h_len) strips += (m + R - 1) / R;
  const uint64_t most_q = (qs->max_len + R - 1) / R;
  // the streams that packed_score builds
  const uint64_t lane = std::max(most_q, 32 * (strips / 2 * residues / slots / (2 * longest)));
  uint64_t K = std::min<uint64_t>(qs->n, (strips + lane - 1) / lane);
  const uint64_t units = dual ? K : (K + 1) / 2;
  if (!dual) K = 2 * units;
  const uint64_t ns = std::max(most_q, (strips + K - 1) / K);
  const uint64_t limit = ns * units * residues / halves / slots * 3 / 5;
  double work = 0;
  uint32_t g = 0;
  for (int most = 32; most >= WAVE_FEW_LANES; most /= 2) {
    const uint64_t past = most > WAVE_FEW_LANES ? wave_longest(ns, most, limit) : 0;
    const uint64_t G = wave_lanes(ns, most, (uint64_t)n_groups * GROUP / halves * units, slots);
    uint64_t cols = 0;
    for (; g < n_groups && db->h_glen[g] > past; ++g) cols += (uint64_t)db->h_glen[g] * GROUP;
    work += (double)cols * (double)((ns + G - 1) / G * G);
  }
  work *= (double)units / (double)(halves * 32 * 4 * ctx->sm_count) * (dual ? 1.17 : 1.0);
  const double chain = 2.5 * (double)((ns + 31) / 32) * (double)longest;
  return std::max(work, chain) * (local ? 11 * R + 45 : 8 * R + 66);
}

// Strip rows of the wavefront search: 24 spread a step's hand-over over more
// rows, 16 pad short queries and fill some bands better.  A search whose queries
// fill one band (32 lanes) at 8 rows, and whose lanes fill the chip three times at
// most, lasts about as long as its longest target, so it takes the shortest steps:
// 128 residues against 2,000 targets 0.53 ms (16 rows 0.75, 24 rows 1.01),
// against 12,000 0.91 (1.14, 1.56).  Past one band they lose, 300 residues 1.24
// (0.86, 1.01), and with more lanes too, 16 queries against 2,000 1.48 (1.19,
// 1.18).
int wave_rows(const dsa_ctx* ctx, const dsa_db* db, const dsa_db* qs, uint32_t n_targets, uint64_t residues,
              bool dual, bool local) {
  auto strips = [&](uint32_t R) {
    uint64_t c = 0;
    for (uint32_t m : qs->h_len) c += (m + R - 1) / R;
    return c;
  };
  auto cost = [&](uint32_t R) {
    return wave_cycles(ctx, db, qs, (n_targets + GROUP - 1) / GROUP, residues, R, dual, local);
  };
  const uint64_t lanes = dual ? strips(8) : std::max<uint64_t>((qs->max_len + 7) / 8, (strips(8) + 1) / 2);
  if (lanes <= 32 && lanes * n_targets / (dual ? 2 : 1) <= 3ull * 512 * ctx->sm_count) return 8;
  return cost(16) < cost(24) ? 16 : 24;
}

// Few queries, or one much longer than the rest, leave one of two query
// streams idle: the wavefronts then take two targets a lane.  Such a step reads
// bytes for both residues and joins them (about 1.17 of the time of a step on
// two queries: 32 queries of 200-1,500 against 60,000 targets 80.0 and 93.3 ms).
bool wave_dual(const dsa_db* qs, const Validated& v, bool local, uint32_t max_n, int o, int e) {
  if (!wave_dual_takes(local, qs->max_len, max_n, o, e, v.smax, v.smin)) return false;
  uint64_t sum = 0;
  for (uint32_t m : qs->h_len) sum += m;
  return 2ull * qs->max_len * 10 > sum * 12;
}

// Work on the side stream, joined to the context's stream on every way out of a
// call: the buffers it uses are given back in the order of the context's stream,
// so a call that fails after the fork (an allocation past the budget) must not
// leave it running beside them.
struct SideJoin {
  dsa_ctx* ctx;
  bool open = false;
  int close() {
    if (!open) return DSA_OK;
    open = false;
    DSA_CUDA_TRY(cudaEventRecord(ctx->join_ev, ctx->side));
    DSA_CUDA_TRY(cudaStreamWaitEvent(ctx->stream, ctx->join_ev, 0));
    return DSA_OK;
  }
  ~SideJoin() { close(); }
};

// Packed score pass (int16x2).  Targets of groups longer than `long_thr` go
// to the wavefront kernel, the rest to the inter-sequence kernel; with both,
// the wavefronts run on the side stream.  The results do not depend on
// long_thr, only the time.  Global / semi-global use the end-anchored forms
// of both kernels; searches whose values could pass 16 bits on the wavefronts
// of k_wave.cu take those of k_intra.cu.
int packed_score(dsa_ctx* ctx, dsa_res* res, const dsa_db* db, const dsa_db* qs,
                 const int8_t* d_mat, const int8_t* d_pssm, int A, int o, int e, const Validated& v, Scores out,
                 uint32_t long_thr, int rows, int mode = DSA_LOCAL, uint32_t fe = 15) {
  const bool local = mode == DSA_LOCAL;
  const uint32_t W = (uint32_t)rows;   // strip rows of the inter-sequence kernel
  const uint32_t nq = qs->n, nt = db->n;
  const int R = A + 1;
  std::vector<uint32_t> qorder(nq);
  std::iota(qorder.begin(), qorder.end(), 0u);
  std::stable_sort(qorder.begin(), qorder.end(),
                   [&](uint32_t a, uint32_t b) { return qs->h_len[a] > qs->h_len[b]; });

  // groups whose longest target exceeds the threshold go to the wavefront kernel
  uint32_t g_long = 0;
  while (g_long < db->n_groups && db->h_glen[g_long] > long_thr) ++g_long;
  const uint32_t n_long = std::min<uint32_t>(nt, g_long * GROUP);
  const bool inter = g_long < db->n_groups;
  const bool wave = n_long && wave_takes(local, qs->max_len, db->h_glen[0], o, e, v.smax, v.smin);

  Streams st;
  if (inter) st = build_streams(qs, qorder, W);
  std::vector<StripMeta>& smeta = st.meta;
  std::vector<uint32_t>&s_sbase = st.sbase, &s_ns = st.ns;
  PackedPlan spl;
  spl.R = R;
  spl.rows = rows;
  spl.n_units = (uint32_t)s_ns.size();
  spl.n_strips = (uint32_t)smeta.size();

  const uint32_t blocks = (db->n_groups - g_long + INTER_WARPS - 1) / INTER_WARPS;
  struct Item { uint64_t cost; uint32_t p, g0; };
  std::vector<Item> items;
  items.reserve((size_t)spl.n_units * blocks);
  for (uint32_t u = 0; u < spl.n_units; ++u)
    for (uint32_t b = 0; b < blocks; ++b) {
      const uint32_t g0 = g_long + b * INTER_WARPS;
      items.push_back({(uint64_t)db->h_glen[g0] * s_ns[u], u, g0});
    }
  std::stable_sort(items.begin(), items.end(),
                   [](const Item& a, const Item& b) { return a.cost > b.cost; });
  std::vector<uint32_t> item_words(2 * items.size());
  for (size_t k = 0; k < items.size(); ++k) {
    item_words[2 * k] = items[k].p;
    item_words[2 * k + 1] = items[k].g0;
  }
  InterWork iw;
  iw.n_items = (uint32_t)items.size();
  iw.max_glen = g_long < db->n_groups ? db->h_glen[g_long] : 0;

  // Pair plan for the wavefront kernel: one query per half (sorted neighbours).
  PackedPlan ppl;
  IntraWork xw;
  std::vector<StripMeta> pmeta;
  std::vector<uint32_t> p_sbase, p_ns, long_ids, litem_words;
  uint64_t long_res = 0;
  for (uint32_t li = 0; li < n_long; ++li) long_res += db->h_len[db->h_perm[li]];
  if (n_long && !wave) {
    ppl.R = R;
    ppl.rows = 32;   // the wavefront kernel's lanes take half-strips of 16 rows
    auto strips32 = [&](uint32_t q) { return (qs->h_len[q] + 31u) / 32u; };
    for (uint32_t u = 0; 2 * u < nq; ++u) {
      const uint32_t qa = qorder[2 * u];
      const uint32_t qb = 2 * u + 1 < nq ? qorder[2 * u + 1] : NONE;
      const uint32_t ns_u = std::max(strips32(qa), qb != NONE ? strips32(qb) : 0u);
      p_sbase.push_back((uint32_t)pmeta.size());
      p_ns.push_back(ns_u);
      for (uint32_t st = 0; st < ns_u; ++st)
        pmeta.push_back({qa, st | (st == ns_u - 1 ? LAST : 0u), qb, st | (st == ns_u - 1 ? LAST : 0u)});
    }
    ppl.n_units = (uint32_t)p_ns.size();
    ppl.n_strips = (uint32_t)pmeta.size();
    long_ids.assign(db->h_perm.begin(), db->h_perm.begin() + n_long);
    struct LItem { uint64_t cost; uint32_t li, p; };
    std::vector<LItem> litems;
    litems.reserve((size_t)n_long * ppl.n_units);
    for (uint32_t li = 0; li < n_long; ++li) {
      const uint32_t L = db->h_len[long_ids[li]];
      xw.max_long_len = std::max(xw.max_long_len, L);
      for (uint32_t u = 0; u < ppl.n_units; ++u) litems.push_back({(uint64_t)L * p_ns[u], li, u});
    }
    std::stable_sort(litems.begin(), litems.end(),
                     [](const LItem& a, const LItem& b) { return a.cost > b.cost; });
    litem_words.resize(2 * litems.size());
    for (size_t k = 0; k < litems.size(); ++k) {
      litem_words[2 * k] = litems[k].li;
      litem_words[2 * k + 1] = litems[k].p;
    }
    xw.n_items = (uint32_t)litems.size();
  }
  uint64_t qsum = 0;
  for (uint32_t x : qs->h_len) qsum += x;
  if (res) {
    res->phase_cells[PH_INTRA] = qsum * long_res;
    res->phase_cells[PH_INTER] = qsum * (db->n_res - long_res);
  }

  // end-anchored strips: the padding rows above a query reproduce row 0
  // (S + o = 0 against the boundary -(o + (j-1)e), o against a free begin)
  const int tpad = (mode == DSA_SEMIGLOBAL && (fe & DSA_FREE_T_BEGIN)) ? o : 0;
  // long targets beside an inter-sequence launch run on the side stream: the
  // two kernels write disjoint targets' results
  cudaStream_t ls = ctx->stream;
  DevBuf d_pmeta, d_pbase, d_pns, d_pprof, d_long, d_litems;
  SideJoin join{ctx};   // before the buffers above and the caller's scores are given back
  if (n_long && inter) {
    ls = ctx->side;
    DSA_CUDA_TRY(cudaEventRecord(ctx->fork_ev, ctx->stream));
    DSA_CUDA_TRY(cudaStreamWaitEvent(ctx->side, ctx->fork_ev, 0));
    join.open = true;
  }
  if (wave) {
    bool dual = wave_dual(qs, v, local, db->h_glen[0], o, e);
    int wr = wave_rows(ctx, db, qs, n_long, long_res, dual, local);
    // two targets a lane halve the work but not the longest target's chain: not
    // where the work, as strip columns per lane of the chip, is the shorter (one
    // query of 300 residues against 2,000 targets, global, 0.70 and 0.96 ms, of
    // 700 against 50,000 4.0 and 2.5)
    if (dual) {
      const uint64_t steps = (uint64_t)((qs->max_len + wr - 1) / wr) * long_res / (ctx->sm_count * 512ull);
      if (steps * 4 < 3ull * db->h_glen[0]) {
        dual = false;
        wr = wave_rows(ctx, db, qs, n_long, long_res, dual, local);
      }
    }
    // longer streams waste fewer lanes and balance the halves better, until the
    // longest target's pass over a unit would take half the launch: each of the
    // chip's lanes has total / lanes strip columns to compute, the longest
    // target's 32 lanes one per column and band
    uint64_t strips = 0;
    for (uint32_t m : qs->h_len) strips += (m + wr - 1) / wr;
    const uint64_t share = strips / 2 * long_res / ((uint64_t)ctx->sm_count * 512);
    const Streams ws =
        build_streams(qs, qorder, (uint32_t)wr, 32 * (share / (2ull * db->h_glen[0])), dual);
    phase_begin(res, PH_INTRA, ls);
    DSA_TRY(launch_wave_search(ctx, ls, db, qs, d_mat, d_pssm, A, mode, fe, o, e, v.smax, v.smin, wr,
                               dual, ws.meta, ws.sbase, ws.ns, n_long, long_res, out));
    phase_end(res, PH_INTRA, ls);
  } else if (n_long) {
    DSA_TRY(upload(ctx, d_pmeta, pmeta));
    DSA_TRY(upload(ctx, d_pbase, p_sbase));
    DSA_TRY(upload(ctx, d_pns, p_ns));
    DSA_TRY(upload(ctx, d_long, long_ids));
    DSA_TRY(upload(ctx, d_litems, litem_words));
    DSA_TRY(d_pprof.alloc(ctx, (size_t)ppl.n_strips * R * ppl.pitch * sizeof(uint32_t)));
    ppl.d_meta = d_pmeta.as<StripMeta>();
    ppl.d_sbase = d_pbase.as<uint32_t>();
    ppl.d_ns = d_pns.as<uint32_t>();
    ppl.d_prof = d_pprof.as<uint32_t>();
    xw.d_long_ids = d_long.as<uint32_t>();
    xw.d_items = d_litems.as<uint32_t>();
    DSA_TRY(launch_strip_profile(ctx, qs, d_mat, d_pssm, A, o, ppl, !local, tpad));
    if (inter) {   // the uploads and the profile above
      DSA_CUDA_TRY(cudaEventRecord(ctx->fork_ev, ctx->stream));
      DSA_CUDA_TRY(cudaStreamWaitEvent(ctx->side, ctx->fork_ev, 0));
    }
    phase_begin(res, PH_INTRA, ls);
    DSA_TRY(launch_intra_glob16(ctx, ls, db, qs, ppl, xw, mode, fe, o, e, v.smax, v.smin, out, nt));
    phase_end(res, PH_INTRA, ls);
  }
  if (inter) {
    DevBuf d_smeta, d_sbase, d_sns, d_sprof, d_items;
    DSA_TRY(upload(ctx, d_smeta, smeta));
    DSA_TRY(upload(ctx, d_sbase, s_sbase));
    DSA_TRY(upload(ctx, d_sns, s_ns));
    DSA_TRY(upload(ctx, d_items, item_words));
    DSA_TRY(d_sprof.alloc(ctx, (size_t)spl.n_strips * R * spl.pitch * sizeof(uint32_t)));
    spl.d_meta = d_smeta.as<StripMeta>();
    spl.d_sbase = d_sbase.as<uint32_t>();
    spl.d_ns = d_sns.as<uint32_t>();
    spl.d_prof = d_sprof.as<uint32_t>();
    iw.d_items = d_items.as<uint32_t>();
    const bool sum = sum_fits(local, qs->max_len, iw.max_glen, o, e, v.smax, v.smin);
    DSA_TRY(sum ? launch_strip_profile(ctx, qs, d_mat, d_pssm, A, local ? o + e : 2 * e, spl, !local,
                                       2 * e - (tpad ? 0 : o), true)
                : launch_strip_profile(ctx, qs, d_mat, d_pssm, A, o, spl, !local, tpad));
    phase_begin(res, PH_INTER);
    if (local)
      DSA_TRY(launch_inter_local16(ctx, db, spl, iw, o, e, v.smax, sum, out, nt));
    else
      DSA_TRY(launch_inter_glob16(ctx, db, qs, spl, iw, mode, fe, o, e, v.smax, v.smin, sum, out, nt));
    phase_end(res, PH_INTER);
  }
  return join.close();
}

// Targets longer than this go to the wavefronts when nothing is tuned or
// forced.  The inter-sequence kernel is the faster one where targets abound
// (32 queries of 64-5,000 against 500,000 targets: 6,900 against 6,100
// GCUPS), but a thread there works through its target alone: one column of a
// 28-row strip takes about 1,400 cycles with 16 warps per SM, so its longest
// item must stay well below the launch (a quarter of it).  5 queries of 60-700
// against 60,000 targets took 23.3 ms with a threshold of 4,096, 8.6 with
// 1,024 and 7.2 on the wavefronts alone; 0 where little would be left for the
// inter-sequence kernel.
uint32_t model_threshold(const dsa_db* db, const dsa_db* qs, const Validated& v, bool local, int o, int e) {
  // the inter-sequence kernel would leave one of its two streams idle
  if (wave_dual(qs, v, local, db->h_glen[0], o, e)) return 0;
  uint64_t strips = 0, longest = 1;
  for (uint32_t m : qs->h_len) {
    const uint64_t n = (m + INTER_ROWS - 1) / INTER_ROWS;
    strips += n;
    longest = std::max(longest, n);
  }
  const uint64_t pairs = std::max(longest, strips / 2);   // packed strips
  const double warp_cols = (double)pairs * (double)db->n_res / 32.0;
  const double total = warp_cols * 344.0 / 608.0;   // cycles at full rate
  const double thr = 0.25 * total / ((double)longest * 1378.0);
  const uint32_t t = (uint32_t)std::min(thr, 1e9);
  uint64_t left = 0;   // residues the inter-sequence kernel would get
  for (uint32_t g = db->n_groups; g-- > 0 && db->h_glen[g] <= t;) left += (uint64_t)db->h_glen[g] * GROUP;
  return left * 4 < db->n_res ? 0 : t;
}

// A threshold whose inter-sequence boundary rows (8 bytes per thread and column
// of its longest target) fit: past PLAIN_THRESHOLD columns they may take half of
// what the context can still allocate, so that a long threshold, faster where
// targets abound, is no reason to refuse a call (contigs of up to a million
// residues would take 600 GB; 4,096 columns take at most 2.6).
constexpr uint32_t PLAIN_THRESHOLD = 4096;
uint32_t fit_threshold(dsa_ctx* ctx, const dsa_db* db, uint32_t nq, uint32_t thr) {
  uint32_t g = 0;
  while (g < db->n_groups && db->h_glen[g] > thr) ++g;
  if (g == db->n_groups || db->h_glen[g] <= PLAIN_THRESHOLD) return thr;
  const uint64_t blocks = (db->n_groups - g + INTER_WARPS - 1) / INTER_WARPS;
  const uint64_t ctas = std::min<uint64_t>((nq + 1ull) / 2 * blocks, (uint64_t)inter_blocks_per_sm() * ctx->sm_count);
  const uint64_t column = ctas * INTER_WARPS * 32 * sizeof(uint2);
  if (!ctx->budget && column * db->h_glen[g] <= 4ull << 30) return thr;   // asking takes 30 us
  const uint64_t fits = memory_room(ctx) / 2 / column;
  if (db->h_glen[g] <= fits) return thr;
  return (uint32_t)std::max<uint64_t>(PLAIN_THRESHOLD, fits);
}

// Strip rows forced by DSA_INTER_ROWS (0: let the tuner choose).
int forced_rows() {
  if (const char* env = getenv("DSA_INTER_ROWS")) {
    const int r = atoi(env);
    if (r == INTER_ROWS || r == INTER_ROWS_SHORT) return r;
  }
  return 0;
}

// The packed pass with the autotuned kernel variant (strip rows) and
// long-target threshold.
int run_packed_tuned(dsa_ctx* ctx, dsa_res* res, const dsa_db* db, const dsa_db* qs,
                     const int8_t* d_mat, const int8_t* d_pssm, int A, int o, int e,
                     const Validated& v, Scores out, int mode, uint32_t fe) {
  const bool local = mode == DSA_LOCAL;
  const int rows_forced = forced_rows();
  const char* thr_env = getenv("DSA_LONG_THRESHOLD");
  const uint32_t thr_forced = thr_env ? (uint32_t)strtoul(thr_env, nullptr, 10) : 0;
  auto run = [&](dsa_res* r, uint32_t thr, int rows) {
    return packed_score(ctx, r, db, qs, d_mat, d_pssm, A, o, e, v, out, thr, rows, mode, fe);
  };
  const char* mode_env = getenv("DSA_AUTOTUNE");
  const std::string tmode = mode_env ? mode_env : "cache";
  const int rows_default = rows_forced ? rows_forced : INTER_ROWS;
  auto fit = [&](uint32_t thr) { return fit_threshold(ctx, db, qs->n, thr); };
  const uint32_t thr_default = thr_env ? thr_forced : fit(model_threshold(db, qs, v, local, o, e));
  if (tmode == "off" || (rows_forced && thr_env))
    return run(res, thr_default, rows_default);
  // workload shape key: GPU, driver, the form of the wavefronts (summed, two
  // targets a lane, wrapping, or k_intra.cu's kernel) and, in eighths, how much of
  // the inter-sequence kernel's 28-row and the wavefronts' 16-row strips the
  // queries fill, mode, alphabet, and log2 bins of the query count, query
  // residues, longest query, target count, database residues and longest target
  uint64_t qres = 0;
  uint32_t qmax = 0;
  for (uint32_t x : qs->h_len) { qres += x; qmax = std::max(qmax, x); }
  cudaDeviceProp prop;
  DSA_CUDA_TRY(cudaGetDeviceProperties(&prop, ctx->device));
  int drv = 0;
  cudaDriverGetVersion(&drv);
  const uint32_t longest = db->h_glen[0];
  const char form = wave_dual(qs, v, local, longest, o, e)                          ? 'd'
                    : sum_fits(local, qs->max_len, longest, o, e, v.smax, v.smin)   ? 's'
                    : wave_takes(local, qs->max_len, longest, o, e, v.smax, v.smin) ? 'w'
                                                                                    : 'i';
  auto eighths = [&](uint32_t R) {
    uint64_t rows = 0;
    for (uint32_t m : qs->h_len) rows += (m + R - 1) / R * R;
    return (unsigned)std::min<uint64_t>(99, 8 * rows / qres);
  };
  char key[512];
  snprintf(key, sizeof key, "%s|sm%d|drv%d|wave %c%u.%u|%s|A%d|q%d|qr%d|qm%d|t%d|tr%d|L%d", prop.name,
           ctx->sm_count, drv, form, eighths(INTER_ROWS), eighths(16), local ? "local" : (mode == DSA_GLOBAL ? "global" : "semi"), A,
           ilog2_bin(qs->n), ilog2_bin(qres), ilog2_bin(qmax), ilog2_bin(db->n),
           ilog2_bin(db->n_res), ilog2_bin(db->max_len));
  const std::string key_thr = std::string(key) + "|thr", key_rows = std::string(key) + "|rows";
  Tuner& t = tuner();
  {
    std::lock_guard<std::mutex> lk(t.mu);
    const std::string path = tune_cache_path();
    if (!t.loaded || path != t.path) tune_load(t, path);   // first use, or another file
    auto it_r = t.cache.find(key_rows);
    auto it_t = t.cache.find(key_thr);
    if (tmode != "retune" && it_r != t.cache.end() && it_t != t.cache.end())
      return run(res, thr_env ? thr_forced : fit(it_t->second),
                 rows_forced ? rows_forced : (int)it_r->second);
  }
  if (!ctx->tune)   // contexts that must not spend calls on tuning (serving workers)
    return run(res, thr_default, rows_default);
  std::map<std::pair<uint32_t, int>, double> timed;   // (long groups, rows) -> ms
  auto groups_over = [&](uint32_t thr) {
    uint32_t g = 0;
    while (g < db->n_groups && db->h_glen[g] > thr) ++g;
    return g;
  };
  cudaEvent_t ev0, ev1;
  DSA_CUDA_TRY(cudaEventCreate(&ev0));
  DSA_CUDA_TRY(cudaEventCreate(&ev1));
  int rc = DSA_OK;
  auto measure = [&](uint32_t thr, int rows) -> double {
    const auto k = std::make_pair(groups_over(thr), rows);
    auto it = timed.find(k);
    if (it != timed.end()) return it->second;
    // Short passes run twice, one alone being off by more than 3% at times; the first
    // of a shape also when it is longer, because it maps scratch and loads kernels,
    // and whatever was timed second had won by that.
    const float twice = timed.empty() ? 500.f : 50.f;
    float best_ms = 0.f;
    for (int pass = 0; pass < 2 && rc == DSA_OK && (pass == 0 || best_ms < twice); ++pass) {
      float ms = 0.f;
      if (cudaEventRecord(ev0, ctx->stream) != cudaSuccess) rc = DSA_ERR_CUDA;
      if (rc == DSA_OK) rc = run(nullptr, thr, rows);
      if (rc == DSA_OK && cudaEventRecord(ev1, ctx->stream) != cudaSuccess) rc = DSA_ERR_CUDA;
      if (rc == DSA_OK && cudaEventSynchronize(ev1) != cudaSuccess) rc = DSA_ERR_CUDA;
      if (rc == DSA_OK) cudaEventElapsedTime(&ms, ev0, ev1);
      best_ms = pass ? std::min(best_ms, ms) : ms;
    }
    timed[k] = best_ms;
    return best_ms;
  };
  // 1. the kernel variant (strip rows) at the default threshold, or, where that
  //    leaves the inter-sequence kernel no group, at the plain one (8 queries of 32
  //    against 150,000 targets: 4.5 ms on the wavefronts, 3.8 on 20-row strips); a
  //    switch from the default needs a gain of at least 2%
  int best_rows = rows_default;
  uint32_t best = thr_default;
  double best_ms = measure(thr_default, best_rows);
  const uint32_t thr_inter =
      thr_env || groups_over(thr_default) < db->n_groups ? thr_default : fit(PLAIN_THRESHOLD);
  if (!rows_forced && groups_over(thr_inter) < db->n_groups) {
    const double ms = measure(thr_inter, INTER_ROWS_SHORT);
    if (ms < 0.98 * best_ms) { best_ms = ms; best = thr_inter; best_rows = INTER_ROWS_SHORT; }
  }
  // 2. the long-target threshold: every target on the wavefronts, then a local
  //    search from the best so far by factors of 4 in each direction while it
  //    improves; thresholds that move the same groups as the last one are skipped
  if (!thr_env) {
    if (best) {
      const double ms = measure(0, best_rows);
      if (ms < 0.98 * best_ms) { best_ms = ms; best = 0; }
    }
    const uint32_t from = best ? best : thr_default;
    const uint64_t start = std::max<uint32_t>(from, 1024);
    for (int dir = -1; dir <= 1 && rc == DSA_OK; dir += 2) {
      uint64_t cur = start;
      uint32_t last_g = groups_over(from);
      for (int step = 0; step < 12 && rc == DSA_OK; ++step) {
        const uint64_t nx = dir < 0 ? cur / 4 : cur * 4;
        const uint32_t thr = (dir > 0 && nx >= db->max_len) ? UINT32_MAX : (uint32_t)nx;
        cur = nx;
        const uint32_t g = groups_over(thr);
        if (g == last_g || g == db->n_groups) {
          if (thr == 0 || thr == UINT32_MAX || g == db->n_groups) break;
          continue;
        }
        last_g = g;
        if (fit(thr) != thr) break;
        const double ms = measure(thr, best_rows);
        if (ms < 0.98 * best_ms) {
          best_ms = ms;
          best = thr;
        } else {
          break;
        }
        if (thr == 0 || thr == UINT32_MAX) break;
      }
    }
  }
  cudaEventDestroy(ev0);
  cudaEventDestroy(ev1);
  if (rc) {
    set_error("autotune: %s", cudaGetErrorString(cudaGetLastError()));
    return rc;
  }
  {
    std::lock_guard<std::mutex> lk(t.mu);
    if (!rows_forced) t.cache[key_rows] = (uint32_t)best_rows;
    if (!thr_env) t.cache[key_thr] = best;
    tune_store(t);
  }
  // the final pass with the chosen variant records the phase timings and cells
  return run(res, best, best_rows);
}

}  // namespace

bool tuner_get(const std::string& key, uint32_t* val) {
  Tuner& t = tuner();
  std::lock_guard<std::mutex> lk(t.mu);
  const std::string path = tune_cache_path();
  if (!t.loaded || path != t.path) tune_load(t, path);
  const char* mode_env = getenv("DSA_AUTOTUNE");
  if (mode_env && std::string(mode_env) == "retune") return false;
  auto it = t.cache.find(key);
  if (it == t.cache.end()) return false;
  *val = it->second;
  return true;
}

void tuner_put(const std::string& key, uint32_t val) {
  Tuner& t = tuner();
  std::lock_guard<std::mutex> lk(t.mu);
  t.cache[key] = val;
  tune_store(t);
}

std::string tuner_shape_prefix(dsa_ctx* ctx) {
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, ctx->device) != cudaSuccess) {
    cudaGetLastError();
    return "?";
  }
  int drv = 0;
  cudaDriverGetVersion(&drv);
  char key[320];
  snprintf(key, sizeof key, "%s|sm%d|drv%d", prop.name, ctx->sm_count, drv);
  return key;
}

int tuner_bin(uint64_t x) { return ilog2_bin(x); }

// Score pass for all queries x all targets.
int score_all_vs_all(dsa_ctx* ctx, dsa_res* res, const dsa_db* db, const dsa_db* qs, int mode,
                     uint32_t fe, const int8_t* d_mat, const int8_t* d_pssm, int A, int o, int e, const Validated& v,
                     uint32_t flags, Scores out, uint64_t* n_rerun) {
  const uint32_t nq = qs->n, nt = db->n;
  // int16x2 lanes: local with the saturation flag; global and semi-global
  // with the range flags of the end-anchored kernel (both reruns exact)
  const bool packed = !(flags & (DSA_FORCE_INT32 | DSA_PLAIN_FORM)) &&
                      (mode == DSA_LOCAL ? o >= 1 : true) && o + e <= 4096 &&
                      v.smax + o < 8192 && v.smin > -8192;
  *n_rerun = 0;
  if (!packed) {
    // exact int32: one launch per query over every target (input order)
    std::vector<uint64_t> poff(nq);
    uint64_t words = 0;
    for (uint32_t q = 0; q < nq; ++q) {
      poff[q] = words;
      words += (uint64_t)A * ((qs->h_len[q] + 7u) & ~7u);
    }
    DevBuf d_prof, d_poff, d_scr;
    DSA_TRY(d_prof.alloc(ctx, words * sizeof(int32_t)));
    DSA_TRY(upload(ctx, d_poff, poff));
    DSA_TRY(launch_profile_int32(ctx, qs, d_mat, d_pssm, A, d_prof.as<int32_t>(), d_poff.as<uint64_t>()));
    DSA_TRY(d_scr.alloc(ctx, db->n_res * sizeof(int2)));
    if (res) {
      uint64_t qsum = 0;
      for (uint32_t x : qs->h_len) qsum += x;
      res->phase_cells[PH_INT32] += qsum * db->n_res;
    }
    phase_begin(res, PH_INT32);
    for (uint32_t q = 0; q < nq; ++q)
      DSA_TRY(launch_generic_int32(ctx, db, qs, d_prof.as<int32_t>(), d_poff.as<uint64_t>(),
                                   nullptr, nt, q, d_scr.as<int2>(), mode, fe, o, e, 0, out));
    phase_end(res, PH_INT32);
    return DSA_OK;
  }

  // ---- packed path ----
  DSA_TRY(ensure_interleaved(ctx, db));
  DSA_TRY(run_packed_tuned(ctx, res, db, qs, d_mat, d_pssm, A, o, e, v, out, mode, fe));

  // ---- exact int32 rerun of saturated pairs ----
  const uint64_t n_out = (uint64_t)nq * nt;
  const uint32_t cap = (uint32_t)std::min<uint64_t>(n_out, 1u << 22);
  DevBuf d_list;
  DSA_TRY(d_list.alloc(ctx, (size_t)cap * sizeof(uint32_t)));
  uint32_t* d_count = ctx->d_counters + 1;
  DSA_CUDA_TRY(cudaMemsetAsync(d_count, 0, sizeof(uint32_t), ctx->stream));
  DSA_TRY(launch_collect_flags(ctx, out.flag, n_out, d_list.as<uint32_t>(), cap, d_count));
  uint32_t count = 0;
  DSA_CUDA_TRY(cudaMemcpyAsync(&count, d_count, sizeof(count), cudaMemcpyDeviceToHost, ctx->stream));
  DSA_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  *n_rerun = count;
  if (count == 0) return DSA_OK;
  std::vector<PairJob> jobs;
  if (count > cap) {
    // too many to list: rerun everything in int32
    return score_all_vs_all(ctx, res, db, qs, mode, fe, d_mat, d_pssm, A, o, e, v, flags | DSA_FORCE_INT32,
                            out, n_rerun);
  }
  std::vector<uint32_t> list(count);
  DSA_CUDA_TRY(cudaMemcpyAsync(list.data(), d_list.p, count * sizeof(uint32_t),
                               cudaMemcpyDeviceToHost, ctx->stream));
  DSA_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  std::sort(list.begin(), list.end());
  jobs.resize(count);
  uint64_t scr = 0;
  for (uint32_t k = 0; k < count; ++k) {
    const uint32_t q = list[k] / nt, t = list[k] % nt;
    jobs[k] = {db->h_off[t], scr, q, db->h_len[t], list[k], 0};
    scr += db->h_len[t];
  }
  std::vector<uint64_t> poff(nq);
  uint64_t pw = 0;
  for (uint32_t q = 0; q < nq; ++q) {
    poff[q] = pw;
    pw += (uint64_t)A * ((qs->h_len[q] + 7u) & ~7u);
  }
  DevBuf d_prof32, d_poff32, d_jobs, d_scr;
  DSA_TRY(d_prof32.alloc(ctx, pw * sizeof(int32_t)));
  DSA_TRY(upload(ctx, d_poff32, poff));
  DSA_TRY(launch_profile_int32(ctx, qs, d_mat, d_pssm, A, d_prof32.as<int32_t>(), d_poff32.as<uint64_t>()));
  DSA_TRY(upload(ctx, d_jobs, jobs));
  DSA_TRY(d_scr.alloc(ctx, scr * sizeof(int2)));
  phase_begin(res, PH_INT32);
  DSA_TRY(launch_generic_int32(ctx, db, qs, d_prof32.as<int32_t>(), d_poff32.as<uint64_t>(),
                               d_jobs.as<PairJob>(), count, 0, d_scr.as<int2>(), mode, fe, o, e, 1,
                               out));
  phase_end(res, PH_INT32);
  return DSA_OK;
}

}  // namespace dsa
