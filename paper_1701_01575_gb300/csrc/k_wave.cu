// Database search on wavefronts, packed int16x2 (the score pass of the map
// phase, Sec. II.B.1; DSW / DNW / DSG of Sec. II.C.2): G lanes (4 to 32, a
// power of two) sweep one target against a stream of query strips.
//
// Layout.  As in the inter-sequence kernel the two 16-bit halves of every
// register follow two balanced streams of queries, cut into strips of R rows.
// Lane k of a group holds strip b G + k of the unit in band b and works on
// target column s - k at step s; H and F of a strip's bottom row reach the
// next strip by one shuffle each, one step later.  Only the last strip of a
// band goes through memory (a boundary row per group), every G R rows instead
// of every strip.  A CTA's 8 warps work on neighbouring targets of the length
// order and share the band's query profile in shared memory: 16-byte words
// [residue][row quad][strip], so the lanes of a quarter-warp read different
// banks whatever residues they hold.  Short targets take few lanes (fewer
// steps to fill and drain), the longest ones 32.
//
// Cells.  Values are stored unsigned with a bias B, so that no 16-bit half
// leaves [0, 2^16) and sums are plain 32-bit additions that carry nothing
// between the halves; the profile's packed words are integer sums
// (hi << 16) + lo for the same reason.
//   Local: e j is added to every value of column j, so that E is
//   max(E, H - o + e, floor) with the floor 0 as the third operand:
//     x = Ho_diag + (S + o + e);  H = max(x, E, F);  Ho = H - o;
//     F' = max(F - e, Ho);  E' = max(E, Ho + e, floor of column j + 1)
//   three maxima on the half-rate pipe and three sums, against four and one.
//   Long targets, whose e j would pass 16 bits, take the form of the other
//   local kernels (no e j; maxima that wrap alone).
//   Global and semi-global: e (i + j) is added, and E and F of the next cell
//   are max(H - o + e, E) and max(H - o + e, F): three maxima and one sum.
//   Launches whose scores or gaps could pass 16 bits stay on the kernels of
//   k_intra.cu, so nothing is flagged here.
// Two targets a lane (DUAL).  One query, or one much longer than the rest,
// would leave one stream and so half of every register idle.  Such searches
// follow one stream of all queries, and the halves hold neighbouring targets of
// the length order.  Their columns hold different residues, so the profile is a
// byte per (residue, row), lifted by K to 0..127: two loads give 16 rows of both
// halves and one byte permute a packed cell joins them; K is taken off in the
// same addition.  A step costs about 1.17 of the other form's.  One query
// against 50,000 targets: of 700 residues, local, 4.7 -> 3.0 ms, of 2,000, 13.2
// -> 9.1, global 11.1 -> 7.4; of 128 against 200,000 3.4 -> 2.2.
// Lanes start one after another: before a target's first column they hold the
// padding residue, under which a strip's column-0 state is a fixed point.
//
// Boundary rows.  Lane 0 reads the band above one column ahead of its use.  A
// global step of 16 rows is shorter than that load takes, and the compiler
// waits for it in every step (776 of 1,440 cycles, long scoreboard), so there
// lanes 0 to 3 load the next block's four columns a block ahead and hand them
// over by two shuffles a step: 24 queries of 175 against 20,000 targets, global,
// 12.2 -> 6.3 ms, 7 of 90-1,100 against 50,000 with 16 rows forced 19.6 -> 6.9.
// Steps of 24 rows and local ones are long enough (0 to 7% slower that way), and
// 8 rows are for searches of one band (6% slower).
//
// End cells.  Local: a column maximum above the best of the strip's query so
// far (as known to the lane: shared along the query's lanes every 32 steps)
// parks the column in shared memory; per band the lanes of a query are
// reduced under (score desc, j asc, i asc), the winner looks its row up and
// merges with the earlier bands' result.  Global and semi-global: as in the
// inter-sequence kernel (column n parked, row m tracked).
//
// Bound by the ALU pipe; 128 registers keep 16 warps per SM (the local summed form
// on strips of 24 rows spills 12 bytes, 20 with two targets a lane).  Measured (whole
// score pass, before: the inter-sequence kernel with the longest targets on
// the wavefronts of k_intra.cu): 7 queries of 90-1,100 against 50,011 targets,
// global, 16.1 -> 7.5 ms (7,200 GCUPS); 5 of 60-700 against 60,000, local, 17.1
// -> 5.9 ms; 32 of 64-5,000 against 100,000, local, 225.6 -> 225.3 ms.
#include "dsa_internal.cuh"
#include "dpx.cuh"

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

namespace dsa {
namespace {

constexpr int NW = 8;              // warps per CTA
constexpr int NT = NW * 32;
constexpr int PLANE = 512;         // bytes of one row quad of 32 strips
constexpr int MIN_WARPS = 2;       // busy warps per CTA of spread launches and longest targets
enum Form { LOCAL_SUM = 0, LOCAL_WRAP = 1, GLOBAL_SUM = 2 };

// Targets first .. first + count of the length order against one unit, `G`
// lanes a target (or two), CTA items of `warps` * 32 / G such groups.
struct Segment {
  uint32_t unit, first, count, item0;
  int32_t G, warps;
};

struct WaveArgs {
  const uint8_t* tcodes;
  const uint64_t* toff;
  const uint32_t* tlen;
  const uint32_t* perm;            // length order -> target id
  const uint32_t* prof;            // [strip][residue][R] packed (DUAL: bytes)
  const StripMeta* meta;
  const uint32_t* sbase;
  const uint32_t* nstrips;
  const uint32_t* qlen;
  int A, o, e, mode, bias, T;
  int K;                           // DUAL: what the profile's bytes have too much
  uint32_t fe;
  uint32_t pad_word;               // profile word (DUAL: 4 bytes) of strips past a unit's end
  const Segment* segs;
  uint32_t n_segs, n_items;
  unsigned long long* counter;     // CTAs started << 32 | items taken
  uint2* scratch;
  const uint64_t* slot;            // first boundary cell of the k-th CTA to start
  Scores out;
  uint32_t n_out_t;
};

// Cells of a boundary row: whole 128-byte lines, none shared by two lane groups.
__host__ __device__ inline uint32_t boundary_row(uint32_t n) { return (n + 15) & ~15u; }

template <int FORM, int R, bool DUAL>
__global__ void __launch_bounds__(NT, 2) k_wave(const WaveArgs A) {
  static_assert(!DUAL || FORM != LOCAL_WRAP, "two targets a lane: summed forms");
  constexpr bool LOCAL = FORM != GLOBAL_SUM;
  constexpr bool SUM = FORM != LOCAL_WRAP;
  constexpr unsigned FULL = 0xFFFFFFFFu;
  constexpr uint32_t BIAS2 = 0x80008000u;
  constexpr int RS = DUAL ? 32 * R : R / 4 * PLANE;   // profile bytes per residue
  constexpr int MIN_SLOTS = DUAL ? 16 : 8;
  constexpr bool BLOCK_IN = !LOCAL && R == 16;        // see "Boundary rows"
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ Segment s_seg;
  __shared__ uint32_t s_tile;
  __shared__ uint64_t s_slot;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // parked columns: local [half][8 rows of 16 bits][thread], others packed
  // [row][thread]
  uint4* const park = reinterpret_cast<uint4*>(smem + (A.A + 1) * RS) + tid;
  uint32_t* const parkw = reinterpret_cast<uint32_t*>(smem + (A.A + 1) * RS) + tid;
  const int o = A.o, e = A.e;
  const uint32_t e2 = (uint32_t)e * 0x10001u, o2 = (uint32_t)o * 0x10001u;
  const uint32_t neg_e2 = pack2(-e, -e), c2 = pack2(e - o, e - o);
  const uint32_t mo2 = pack2(-o, -o) ^ BIAS2, K2 = (uint32_t)A.K * 0x10001u;
  const bool sg = A.mode == DSA_SEMIGLOBAL;
  const bool qb_free = sg && (A.fe & DSA_FREE_Q_BEGIN), qe_free = sg && (A.fe & DSA_FREE_Q_END);
  const bool tb_free = sg && (A.fe & DSA_FREE_T_BEGIN), te_free = sg && (A.fe & DSA_FREE_T_END);
  auto row0 = [&](int j) { return (j == 0 || tb_free) ? 0 : -(o + (j - 1) * e); };
  uint2* scr_cta = nullptr;           // the CTA's boundary rows (two targets a lane: no registers left)
  uint32_t held = NONE;               // first strip and group size of the profile in place

  for (bool first = true;; first = false) {
    __syncthreads();
    if (tid == 0) {
      const unsigned long long got = atomicAdd(A.counter, first ? (1ull << 32) + 1 : 1ull);
      const uint32_t item = (uint32_t)got;
      if (first) s_slot = A.slot[got >> 32];
      if (item >= A.n_items) {
        s_tile = NONE;
      } else {
        uint32_t lo = 0, hi = A.n_segs;   // the last segment starting at or before the item
        while (hi - lo > 1) {
          const uint32_t mid = (lo + hi) / 2;
          if (A.segs[mid].item0 <= item) lo = mid;
          else hi = mid;
        }
        s_seg = A.segs[lo];
        s_tile = item - s_seg.item0;
      }
    }
    __syncthreads();
    if (s_tile == NONE) break;
    if (first) scr_cta = A.scratch + s_slot;
    const int G = s_seg.G, k = lane & (G - 1);
    const uint32_t ns = A.nstrips[s_seg.unit], sb = A.sbase[s_seg.unit];
    const uint32_t tile0 = s_tile * (s_seg.warps * 32 / G), group = warp * (32 / G) + lane / G;
    const uint32_t in_seg = (tile0 + group) * (DUAL ? 2 : 1);
    // boundary rows are as long as the item's longest target, its first
    const uint32_t row = (int)ns > G ? boundary_row(A.tlen[A.perm[s_seg.first + tile0 * (DUAL ? 2 : 1)]]) : 0;
    // the halves' targets: the same, or (DUAL) neighbours, the longer one first
    const bool valid = in_seg < s_seg.count && warp < s_seg.warps;
    const bool valid2 = DUAL ? valid && in_seg + 1 < s_seg.count : valid;
    uint32_t id = 0, id2 = 0;
    int n = 0, n2 = 0;
    const uint8_t *t = A.tcodes, *t2 = A.tcodes;
    if (valid) {
      id = A.perm[s_seg.first + in_seg];
      n = (int)A.tlen[id];
      t = A.tcodes + A.toff[id];
    }
    if (!DUAL) {
      id2 = id;
      n2 = n;
    } else if (valid2) {
      id2 = A.perm[s_seg.first + in_seg + 1];
      n2 = (int)A.tlen[id2];
      t2 = A.tcodes + A.toff[id2];
    }
    int nmax = n, nmin = n2;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
      nmax = max(nmax, __shfl_xor_sync(FULL, nmax, w));
      nmin = min(nmin, __shfl_xor_sync(FULL, nmin, w));
    }
    const uint32_t sh = 8u * (uint32_t)((uintptr_t)(t - k) & 3), sh2 = 8u * (uint32_t)((uintptr_t)(t2 - k) & 3);
    uint2* const scr = (DUAL ? A.scratch + s_slot : scr_cta) + (uint64_t)group * row;
    const int steps = nmax + G - 1;
    const int nb = ((int)ns + G - 1) / G;

    for (int b = 0; b < nb; ++b) {
      const uint32_t want = (sb + (uint32_t)(b * G)) * 64u + (uint32_t)G;
      if (held != want) {
        __syncthreads();
        // slot x of 8 (DUAL: 16) or more holds strip x mod G: fewer lanes a target
        // read copies
        const int slots = max(G, MIN_SLOTS), lg = 31 - __clz(slots);
        const int total = slots * (A.A + 1) * (DUAL ? R / 8 : R / 4);
        for (int x = tid; x < total; x += NT) {
          const int slot = x & (slots - 1), rest = x >> lg;
          const uint32_t strip = (uint32_t)(b * G + (slot & (G - 1)));
          if (DUAL) {   // 8 rows, into a plane of 16 or (the last 8 rows) of 8 bytes a slot
            constexpr int C = R / 8;
            const int a = rest / C, c = rest - a * C;
            uint2 v = make_uint2(A.pad_word, A.pad_word);
            if (strip < ns)
              v = __ldg(reinterpret_cast<const uint2*>(A.prof + (uint64_t)(sb + strip) * (A.A + 1) * (R / 4)) + rest);
            *reinterpret_cast<uint2*>(smem + a * RS + (R != 8 && c < 2 ? slot * 16 + c * 8 : (R != 8 ? PLANE : 0) + slot * 8)) = v;
            continue;
          }
          uint4 v = make_uint4(A.pad_word, A.pad_word, A.pad_word, A.pad_word);
          if (strip < ns)
            v = __ldg(reinterpret_cast<const uint4*>(A.prof + (uint64_t)(sb + strip) * (A.A + 1) * R) + rest);
          *reinterpret_cast<uint4*>(smem + rest * PLANE + slot * 16) = v;
        }
        __syncthreads();
        held = want;
      }
      const int slot = lane & (max(G, MIN_SLOTS) - 1);
      const uint8_t* const pbase = smem + slot * (DUAL && R == 8 ? 8 : 16);
      StripMeta md{NONE, 0, NONE, 0};
      if ((uint32_t)(b * G + k) < ns) md = A.meta[sb + b * G + k];
      const int ka = (int)(md.ka & ~LAST), kb = (int)(md.kb & ~LAST);
      const uint32_t keep = (ka == 0 ? 0u : 0x0000FFFFu) | (kb == 0 ? 0u : 0xFFFF0000u);
      const bool last_a = (md.ka & LAST) && md.qa != NONE, last_b = (md.kb & LAST) && md.qb != NONE;

      // ---- column-0 state ----
      int j = -k;                    // the lane's column
      uint32_t Ho[R], E[R], diag, sendH, sendF;
      uint32_t flo2 = mo2, fln2 = 0; // local: H = 0 as H - o at column j, the floor of column j + 1
      uint32_t rthr = 0xFFFFFFFFu, rinc = 0;
      int rj_a = 0, rj_b = 0;
      uint32_t hmn = 0;
      if (LOCAL) {
        if (SUM) {
          flo2 = (uint32_t)(A.bias + e * j - o) * 0x10001u;
          fln2 = flo2 + o2 + e2;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          Ho[r] = flo2;
          E[r] = SUM ? fln2 : pack2(NEG16, NEG16) ^ BIAS2;
        }
        diag = sendH = sendF = flo2;
      } else {
        // H of column 0 at padded row i, and F entering row i + 1 there, with
        // e (i + j) added; a half without a query is all padding rows
        const int ma = md.qa != NONE ? (int)A.qlen[md.qa] : 0, mb = md.qb != NONE ? (int)A.qlen[md.qb] : 0;
        const int pa = md.qa != NONE ? (R - ma % R) % R : INT32_MAX;
        const int pb = md.qb != NONE ? (R - mb % R) % R : INT32_MAX;
        auto hv = [&](int i, int p) {
          const int h = (i <= p || qb_free) ? 0 : -(o + (i - p - 1) * e);
          return A.bias + h + e * (i + j);
        };
        auto fv = [&](int i, int p) {
          const int f = (i <= p || qb_free) ? -o : -(o + (i - p) * e);
          return A.bias + f + e * (i + 1 + j);
        };
        const int ba = ka * R, bb = kb * R;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          Ho[r] = pack2(hv(ba + r + 1, pa), hv(bb + r + 1, pb));
          E[r] = add2(Ho[r], c2);
        }
        diag = pack2(hv(ba, pa), hv(bb, pb));
        sendH = Ho[R - 1];
        sendF = pack2(fv(ba + R, pa), fv(bb + R, pb));
        if (te_free && last_a) { rthr = (rthr & 0xFFFF0000u) | (uint32_t)hv(ba + R, pa); rinc |= (uint32_t)e; }
        if (te_free && last_b) { rthr = (rthr & 0x0000FFFFu) | (uint32_t)hv(bb + R, pb) << 16; rinc |= (uint32_t)e << 16; }
      }
      // local: the best this lane has seen per half in this band, the best of
      // its query's earlier bands and, from the last exchange, of its lanes,
      // and the trigger threshold
      int best_a = 0, best_b = 0, bj_a = 0, bj_b = 0;
      uint32_t shared2 = 0, thr2 = 0;
      if (LOCAL && b > 0 && valid) {
        if (ka > k) shared2 = (uint32_t)min(A.out.score[(uint64_t)md.qa * A.n_out_t + id], 0xFFFF);
        if (kb > k && valid2) shared2 |= (uint32_t)min(A.out.score[(uint64_t)md.qb * A.n_out_t + id2], 0xFFFF) << 16;
      }
      auto set_thr = [&]() {   // columns whose maximum reaches the best trigger
        const uint32_t v = __vmaxu2(shared2, pack2(best_a, best_b));
        thr2 = __vsubus2(v, 0x00010001u) + (SUM ? flo2 + o2 : BIAS2);
      };
      if (LOCAL) set_thr();
      const bool hand = b + 1 < nb && k == G - 1;   // the band's bottom row is read again
      uint2 in = make_uint2(0, 0), in_nxt = in;
      if (b > 0 && k < (BLOCK_IN ? min(4, n) : min(1, n))) in_nxt = scr[k];
      if (!BLOCK_IN) in = in_nxt;

      // residues of 4 steps, one block ahead: two aligned words, or (edge) the
      // four bytes with the padding residue outside the target
      auto edge_at = [&](int s0) { return s0 < G - 1 || s0 + 4 > nmin; };
      auto fetch = [&](int s0, const uint8_t* t, int n) -> uint2 {
        const int x = s0 - k;
        if (!edge_at(s0)) {
          const uint32_t* p = reinterpret_cast<const uint32_t*>((uintptr_t)(t + x) & ~(uintptr_t)3);
          return make_uint2(__ldg(p), __ldg(p + 1));
        }
        uint32_t w = 0;
#pragma unroll
        for (int y = 0; y < 4; ++y)
          w |= ((uint32_t)(x + y) < (uint32_t)n ? (uint32_t)__ldg(t + x + y) : (uint32_t)A.A) << (8 * y);
        return make_uint2(w, 0);
      };
      uint2 nxt = fetch(0, t, n), nxt2 = DUAL ? fetch(0, t2, n2) : make_uint2(0, 0);
      for (int s0 = 0; s0 < steps; s0 += 4) {
        const uint32_t r4 = edge_at(s0) ? nxt.x : __funnelshift_r(nxt.x, nxt.y, sh);
        nxt = fetch(s0 + 4, t, n);
        if (BLOCK_IN) {
          in = in_nxt;
          if (b > 0 && k < 4 && s0 + 4 + k < n) in_nxt = scr[s0 + 4 + k];
        }
        uint32_t r4b = 0;
        if (DUAL) {
          r4b = edge_at(s0) ? nxt2.x : __funnelshift_r(nxt2.x, nxt2.y, sh2);
          nxt2 = fetch(s0 + 4, t2, n2);
        }
        if (LOCAL && ((s0 & 31) == 28 || s0 == 4 || s0 == 12)) {
          // the best of the query's lanes: maxima over the lanes above and
          // below that hold the same query, per half
          const int fa = max(0, k - ka), fb = max(0, k - kb);
          uint32_t v = __vmaxu2(shared2, pack2(best_a, best_b));
          for (int w = 1; w < G; w <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, v, w);
            const uint32_t ok = (k - w >= fa ? 0x0000FFFFu : 0u) | (k - w >= fb ? 0xFFFF0000u : 0u);
            const uint32_t d = __shfl_down_sync(FULL, v, w);
            const int fda = __shfl_down_sync(FULL, fa, w), fdb = __shfl_down_sync(FULL, fb, w);
            const uint32_t okd = k + w < G ? (fda <= k ? 0x0000FFFFu : 0u) | (fdb <= k ? 0xFFFF0000u : 0u) : 0u;
            v = max3_2u(v, u & ok, d & okd);
          }
          shared2 = v;
          set_thr();
        }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          ++j;
          uint32_t upH = __shfl_up_sync(FULL, sendH, 1);
          uint32_t upF = __shfl_up_sync(FULL, sendF, 1);
          if (BLOCK_IN) {
            if (b > 0) {
              const int from = (lane & ~(G - 1)) + y;
              const uint32_t h = __shfl_sync(FULL, in.x, from), f = __shfl_sync(FULL, in.y, from);
              upH = k == 0 ? h : upH;
              upF = k == 0 ? f : upF;
            }
          } else if (b > 0 && k == 0) {
            upH = in.x;
            upF = in.y;
            if (j < n) in = scr[j];
          }
          uint32_t bH, bF;   // row 0 at this column, where a query starts
          if (LOCAL) {
            if (SUM) { flo2 += e2; fln2 += e2; thr2 += e2; }
            bH = bF = flo2;
          } else {
            const int v = A.bias + ((tb_free || j <= 0) ? e * j : e - o);
            bH = (uint32_t)v * 0x10001u;
            bF = (uint32_t)(v + e - o) * 0x10001u;
          }
          const uint32_t topH = (upH & keep) | (bH & ~keep);
          uint32_t F = (upF & keep) | (bF & ~keep);
          const uint32_t aoff = ((r4 >> (8 * y)) & 0xFFu) * RS, boff = ((r4b >> (8 * y)) & 0xFFu) * RS;
          const uint8_t* const p = pbase + aoff;
          uint32_t pa[DUAL ? R / 4 : 1], pb[DUAL ? R / 4 : 1];   // DUAL: the rows' bytes of the two residues
          if (DUAL) {
            if (R == 8) {
              const uint2 va = *reinterpret_cast<const uint2*>(p), vb = *reinterpret_cast<const uint2*>(pbase + boff);
              pa[0] = va.x; pa[1] = va.y; pb[0] = vb.x; pb[1] = vb.y;
            } else {
              const uint4 va = *reinterpret_cast<const uint4*>(p), vb = *reinterpret_cast<const uint4*>(pbase + boff);
              pa[0] = va.x; pa[1] = va.y; pa[2] = va.z; pa[3] = va.w;
              pb[0] = vb.x; pb[1] = vb.y; pb[2] = vb.z; pb[3] = vb.w;
            }
            if (R == 24) {
              const uint8_t* const p8 = smem + PLANE + slot * 8;
              const uint2 va = *reinterpret_cast<const uint2*>(p8 + aoff), vb = *reinterpret_cast<const uint2*>(p8 + boff);
              pa[R / 4 - 2] = va.x; pa[R / 4 - 1] = va.y; pb[R / 4 - 2] = vb.x; pb[R / 4 - 1] = vb.y;
            }
          }
          uint32_t d = diag;
          diag = topH;
          uint32_t cm = 0, hprev = 0;
#pragma unroll
          for (int q = 0; q < R / 4; ++q) {
            uint32_t pr[4];
            if (DUAL) {   // the bytes are at most 127: the selector's sign copies are zeros
#pragma unroll
              for (uint32_t u = 0; u < 4; ++u)
                pr[u] = prmt(pa[q], pb[q], u | (8 + u) << 4 | (4 + u) << 8 | (12 + u) << 12) - K2;
            } else {
              const uint4 pv = *reinterpret_cast<const uint4*>(p + q * PLANE);
              pr[0] = pv.x; pr[1] = pv.y; pr[2] = pv.z; pr[3] = pv.w;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int r = q * 4 + u;
              const uint32_t old = Ho[r];
              uint32_t h;
              if (FORM == LOCAL_SUM) {
                h = max3_2u(d + pr[u], E[r], F);
                const uint32_t ho = h - o2;
                F = addmax2u(F, neg_e2, ho);
                E[r] = max3_2u(E[r], ho + e2, fln2);
                Ho[r] = ho;
              } else if (FORM == LOCAL_WRAP) {
                E[r] = addmax2u(E[r], neg_e2, old);
                const uint32_t x = addmax2u(d, pr[u], E[r]);
                h = max3_2u(x, F, BIAS2);
                Ho[r] = h - o2;
                F = addmax2u(F, neg_e2, Ho[r]);
              } else {
                h = max3_2u(d + pr[u], E[r], F);
                E[r] = addmax2u(h, c2, E[r]);
                F = addmax2u(h, c2, F);
                Ho[r] = h;
              }
              d = old;
              if (LOCAL) {
                if (r & 1) cm = max3_2u(cm, hprev, h);
                else hprev = h;
              }
            }
          }
          sendH = Ho[R - 1];
          sendF = F;
          if (b + 1 < nb && hand && (uint32_t)(j - 1) < (uint32_t)n) scr[j - 1] = make_uint2(sendH, sendF);
          if (LOCAL) {
            if (__vmaxu2(cm, thr2) != thr2) {
              const int z = (int)(SUM ? (flo2 & 0xFFFFu) + (uint32_t)o : 0x8000u);   // H = 0
              const int ca = (int)(cm & 0xFFFFu) - z, cb = (int)(cm >> 16) - z;
              // (the other half may have raised the threshold's alarm)
              if (ca > best_a && ca >= (int)(shared2 & 0xFFFFu)) {
#pragma unroll
                for (int r = 0; r < R; r += 8)
                  park[r / 8 * NT] = make_uint4(prmt(Ho[r], Ho[r + 1], 0x5410), prmt(Ho[r + 2], Ho[r + 3], 0x5410),
                                                prmt(Ho[r + 4], Ho[r + 5], 0x5410), prmt(Ho[r + 6], Ho[r + 7], 0x5410));
                best_a = ca; bj_a = j;
              }
              if (cb > best_b && cb >= (int)(shared2 >> 16)) {
#pragma unroll
                for (int r = 0; r < R; r += 8)
                  park[(R + r) / 8 * NT] =
                      make_uint4(prmt(Ho[r], Ho[r + 1], 0x7632), prmt(Ho[r + 2], Ho[r + 3], 0x7632),
                                 prmt(Ho[r + 4], Ho[r + 5], 0x7632), prmt(Ho[r + 6], Ho[r + 7], 0x7632));
                best_b = cb; bj_b = j;
              }
              set_thr();
            }
          } else {
            if (te_free) {
              rthr += rinc;
              if (__vmaxu2(sendH, rthr) != rthr && j >= 1 && j <= n) {
                if ((sendH & 0xFFFFu) > (rthr & 0xFFFFu)) {
                  rthr = (rthr & 0xFFFF0000u) | (sendH & 0xFFFFu);
                  rj_a = j;
                }
                if ((sendH >> 16) > (rthr >> 16) && (!DUAL || j <= n2)) {
                  rthr = (rthr & 0x0000FFFFu) | (sendH & 0xFFFF0000u);
                  rj_b = j;
                }
              }
            }
            if (DUAL) {   // each half at its own column n
              if (j == n) {
                hmn = (hmn & 0xFFFF0000u) | (sendH & 0xFFFFu);
                if (qe_free) {
#pragma unroll
                  for (int r = 0; r < R; ++r) reinterpret_cast<uint16_t*>(parkw + r * NT)[0] = (uint16_t)Ho[r];
                }
              }
              if (j == n2) {
                hmn = (hmn & 0x0000FFFFu) | (sendH & 0xFFFF0000u);
                if (qe_free) {
#pragma unroll
                  for (int r = 0; r < R; ++r) reinterpret_cast<uint16_t*>(parkw + r * NT)[1] = (uint16_t)(Ho[r] >> 16);
                }
              }
            } else if (j == n) {
              hmn = sendH;
              if (qe_free) {
#pragma unroll
                for (int r = 0; r < R; ++r) parkw[r * NT] = Ho[r];
              }
            }
          }
        }
      }

      // ---- the band's results, one half at a time ----
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const uint32_t q = x ? md.qb : md.qa, idx_t = x ? id2 : id;
        const int nx = x ? n2 : n;
        const bool validx = x ? valid2 : valid;
        const int kq = x ? kb : ka;
        const int first = max(0, k - kq);         // the query's first lane in this band
        const bool starts = k - first == kq;      // its first strip is in this band
        const int sh16 = 16 * x;
        if (LOCAL) {
          int s = x ? best_b : best_a, jj = x ? bj_b : bj_a, src = lane;
          for (int w = 1; w < G; w <<= 1) {
            const int s2 = __shfl_down_sync(FULL, s, w), j2 = __shfl_down_sync(FULL, jj, w);
            const int src2 = __shfl_down_sync(FULL, src, w);
            const int f2 = __shfl_down_sync(FULL, first, w);
            const uint32_t q2 = __shfl_down_sync(FULL, q, w);
            // lanes k .. k + w hold the same query: a tie keeps the smaller rows
            if (k + w < G && q2 == q && f2 <= k && (s2 > s || (s2 == s && s2 > 0 && j2 < jj))) {
              s = s2; jj = j2; src = src2;
            }
          }
          const int win = __shfl_sync(FULL, src, (lane & ~(G - 1)) + first);
          if (validx && q != NONE && win == lane) {
            const int bs = x ? best_b : best_a, bj = x ? bj_b : bj_a;
            int bi = 0;
            if (bs > 0) {
              const uint16_t wanted = (uint16_t)(SUM ? bs - o + A.bias + e * bj : bs - o + 0x8000);
              int rr = R - 1;
              for (int r = R - 1; r >= 0; --r)
                if (reinterpret_cast<const uint16_t*>(park + (x * R + r) / 8 * NT)[r & 7] == wanted) rr = r;
              bi = kq * R + rr + 1;
            }
            const uint64_t idx = (uint64_t)q * A.n_out_t + idx_t;
            bool put = starts;
            if (!put && bs > 0) {
              const int os = A.out.score[idx], ot = A.out.t_end[idx];
              put = bs > os || (bs == os && bj - 1 < ot);   // earlier bands hold smaller rows
            }
            if (put) {
              A.out.score[idx] = bs;
              A.out.q_end[idx] = bi - 1;
              A.out.t_end[idx] = bs > 0 ? bj - 1 : -1;
              A.out.flag[idx] = bs > A.T ? 1 : 0;
            }
          }
        } else {
          const int m = q != NONE ? (int)A.qlen[q] : 0, pad = (R - m % R) % R;
          const int base = kq * R;
          // column n (free query end): this strip's real rows, smallest i first
          int cb = INT32_MIN, ci = 0;
          if (qe_free && q != NONE) {
            for (int r = 0; r < R; ++r) {
              const int i = base + r + 1;
              const int v = (int)((parkw[r * NT] >> sh16) & 0xFFFFu) - A.bias - e * (i + nx);
              if (i > pad && v > cb) { cb = v; ci = i - pad; }
            }
          }
          if (qe_free) {
            for (int w = 1; w < G; w <<= 1) {
              const int s2 = __shfl_down_sync(FULL, cb, w), i2 = __shfl_down_sync(FULL, ci, w);
              const int f2 = __shfl_down_sync(FULL, first, w);
              const uint32_t q2 = __shfl_down_sync(FULL, q, w);
              if (k + w < G && q2 == q && f2 <= k && (s2 > cb || (s2 == cb && i2 < ci))) { cb = s2; ci = i2; }
            }
            cb = __shfl_sync(FULL, cb, (lane & ~(G - 1)) + first);
            ci = __shfl_sync(FULL, ci, (lane & ~(G - 1)) + first);
          }
          // the query's last lane in this band writes: the result, or with a
          // free query end column n's best so far
          const bool last = x ? last_b : last_a;
          const int strips = (m + R - 1) / R;
          const bool tail = q != NONE && (last || (k == G - 1 && kq < strips - 1));
          if (validx && tail && (last || qe_free)) {
            const uint64_t idx = (uint64_t)q * A.n_out_t + idx_t;
            if (qe_free) {
              const int ps = starts ? row0(nx) : A.out.score[idx], pi = starts ? 0 : A.out.q_end[idx];
              if (ps >= cb) { cb = ps; ci = pi; }   // earlier rows
            }
            int bs = cb, bi = ci, bj = nx;
            if (last) {
              const int corner = (int)((hmn >> sh16) & 0xFFFFu) - A.bias - e * (base + R + nx);
              if (!qe_free || corner > bs) { bs = corner; bi = m; }
              if (te_free) {
                const int rj = x ? rj_b : rj_a;
                // the threshold holds the best's value at the last step's column
                const int rv = (int)((rthr >> sh16) & 0xFFFFu) - A.bias - e * (base + R + j);
                if (rv > bs || (rv == bs && rj < bj)) { bs = rv; bi = m; bj = rj; }
              }
              A.out.score[idx] = bs;
              A.out.q_end[idx] = bi - 1;
              A.out.t_end[idx] = bj - 1;
              A.out.flag[idx] = 0;
            } else {
              A.out.score[idx] = bs;
              A.out.q_end[idx] = bi;
            }
          }
        }
      }
      __syncwarp();
    }
  }
}

// Profile of every strip: [strip][residue][R] packed words, lo / hi the
// scores of the two halves' rows plus `add`.  Local: rows past a query's end,
// absent queries and the padding residue get a score below any.  End-anchored
// (global, semi-global): rows above a query reproduce row 0.
struct ProfArgs {
  const uint8_t* qcodes;
  const uint64_t* qoff;
  const uint32_t* qlen;
  const StripMeta* meta;
  uint32_t n_strips;
  const int8_t* S;
  const int8_t* P;     // position-specific rows, or null
  int A, R, add, form;
  int pad_row, pad_col, none;   // words' halves: padding rows; padding residue on real rows; below any
  uint32_t* prof;
  bool dual;           // a byte per row, none negative
};
__global__ void k_wave_profile(const ProfArgs W) {
  const uint64_t total = (uint64_t)W.n_strips * (W.A + 1) * W.R;
  for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < total;
       x += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t s = (uint32_t)(x / ((uint64_t)(W.A + 1) * W.R));
    const int a = (int)(x / W.R % (W.A + 1)), r = (int)(x % W.R);
    const StripMeta md = W.meta[s];
    auto val = [&](uint32_t q, uint32_t kq) -> int {
      const bool glob = W.form == GLOBAL_SUM;
      if (q == NONE) return glob ? (a == W.A ? W.add : W.pad_row) : W.none;
      const int m = (int)W.qlen[q];
      const int i = (int)(kq & ~LAST) * W.R + r - (glob ? (W.R - m % W.R) % W.R : 0);
      if (i < 0) return a == W.A ? W.add : W.pad_row;
      if (i >= m || (!glob && a == W.A)) return W.none;
      if (a == W.A) return W.pad_col;
      const uint64_t at = W.qoff[q] + (uint64_t)i;
      return (W.P ? (int)W.P[at * W.A + a] : (int)W.S[W.qcodes[at] * W.A + a]) + W.add;
    };
    const int lo = val(md.qa, md.ka);
    if (W.dual) {
      reinterpret_cast<uint8_t*>(W.prof)[x] = (uint8_t)lo;
      continue;
    }
    const int hi = val(md.qb, md.kb);
    W.prof[x] = W.form == LOCAL_WRAP ? pack2(lo, hi) : ((uint32_t)hi << 16) + (uint32_t)lo;
  }
}

// The form of a local launch, or of a global one (-1: k_intra.cu's kernel).
int wave_form(bool local, int64_t m, int64_t n, int o, int e, int smax, int smin) {
  if (sum_fits(local, m, n, o, e, smax, smin)) return local ? LOCAL_SUM : GLOBAL_SUM;
  return local ? LOCAL_WRAP : -1;
}

}  // namespace

// The stored value of 0 in the summed forms: every value stays above 0 (gaps
// fall 3o below, a lane starts up to 63 columns before its target, the score
// of an absent row is -128).
int sum_bias(bool local, int o, int e, int smin) {
  return local ? 512 + o + 64 * e : 4 * o + 64 * e + std::max(0, -smin) + 256;
}
// Values with e j (local) or e (i + j) added stay inside 16 bits for queries of
// up to m and targets of up to n residues; global: and none could have been
// flagged by the wrapping form's range rules.
bool sum_fits(bool local, int64_t m, int64_t n, int o, int e, int smax, int smin) {
  const int64_t up = (int64_t)std::max(0, smax) * std::min(m, n);
  if (local) return up + e * (n + 64) + sum_bias(true, o, e, smin) + 2ll * (o + e) + 512 < 65536;
  if (up > 32767 - std::max(0, smax)) return false;
  if (4ll * o + (m + n + 2) * e + std::max(0, -smin) + 64 >= 32768) return false;
  return up + e * (m + n + 256) + sum_bias(false, o, e, smin) + 2ll * (o + e) + 512 < 65536;
}

// What makes the bytes of a two-target profile at least 0, and whether they
// then fit 7 bits.
static int wave_dual_K(bool local, int o, int e, int smin) {
  return local ? std::max(0, -(smin + o + e)) : std::max({0, -(smin + 2 * e), o - 2 * e});
}
bool wave_dual_takes(bool local, uint32_t max_m, uint32_t max_n, int o, int e, int smax, int smin) {
  const int add = local ? o + e : 2 * e;
  return sum_fits(local, max_m, max_n, o, e, smax, smin) &&
         std::max(0, smax) + add + wave_dual_K(local, o, e, smin) <= 127;
}

bool wave_takes(bool local, uint32_t max_m, uint32_t max_n, int o, int e, int smax, int smin) {
  return wave_form(local, max_m, max_n, o, e, smax, smin) >= 0;
}

int launch_wave_search(dsa_ctx* ctx, cudaStream_t stream, const dsa_db* db, const dsa_db* qs,
                       const int8_t* d_matrix, const int8_t* d_pssm, int A, int mode, uint32_t fe, int o,
                       int e, int smax, int smin, int rows, bool dual, const std::vector<StripMeta>& meta,
                       const std::vector<uint32_t>& sbase, const std::vector<uint32_t>& ns,
                       uint32_t n_targets, uint64_t residues, Scores out) {
  if (n_targets == 0 || ns.empty()) return DSA_OK;
  const bool local = mode == DSA_LOCAL;
  const uint32_t max_n = db->h_len[db->h_perm[0]];
  const int form = wave_form(local, qs->max_len, max_n, o, e, smax, smin);
  auto pick = [&](auto f) {
    constexpr int F = decltype(f)::value;
    constexpr bool D = F != LOCAL_WRAP;
    if (dual) return rows == 8 ? k_wave<F, 8, D> : rows == 16 ? k_wave<F, 16, D> : k_wave<F, 24, D>;
    return rows == 8 ? k_wave<F, 8, false> : rows == 16 ? k_wave<F, 16, false> : k_wave<F, 24, false>;
  };
  auto kern = form == LOCAL_SUM    ? pick(std::integral_constant<int, LOCAL_SUM>{})
              : form == LOCAL_WRAP ? pick(std::integral_constant<int, LOCAL_WRAP>{})
                                   : pick(std::integral_constant<int, GLOBAL_SUM>{});
  if (form < 0 || (dual && !wave_dual_takes(local, qs->max_len, max_n, o, e, smax, smin)) || (rows != 8 && rows != 16 && rows != 24)) {
    set_error("no wavefront form for this search");
    return DSA_ERR_INVALID_ARG;
  }
  const int halves = dual ? 2 : 1;   // targets per lane group
  auto smem_of = [&](int letters) {
    return (size_t)(letters + 1) * (dual ? 32 * rows : rows / 4 * PLANE) + (size_t)rows * NT * 4;
  };
  const size_t smem = smem_of(A);
  DSA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(MAX_ALPHABET)));
  int per_sm = 0;
  DSA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem));
  const uint32_t ctas = (uint32_t)std::max(1, per_sm) * ctx->sm_count;

  // Lanes per target: as many as the unit has strips, up to 8 (more lanes cost
  // more steps to fill and drain on every target, and more of them idle in a
  // unit's last band; 7 queries of 90-1,100 against 50,011 targets, global:
  // 9.3 ms with up to 16, 8.8 with 8).  A target's chain, its columns times the
  // unit's bands, must stay below 0.6 of the launch, whose length in steps is the
  // strip columns per lane of the chip: longer targets take 16 or 32 lanes (one
  // query of 2,000 against 50,000 targets, two targets a lane: 12.3 ms with 32
  // lanes past 2,048 columns alone, 9.1 so; 2 queries of 100 and 800: 3.8 ms at
  // 0.35, 3.25 at 0.5 and 0.7).  Launches with fewer targets than the chip has
  // room for take as many lanes as they can.
  const uint64_t slots = (uint64_t)ctas * NT;
  uint64_t strip_cols = 0;
  for (uint32_t x : ns) strip_cols += x * residues / halves;
  const uint64_t limit = strip_cols / slots * 3 / 5;
  std::vector<Segment> segs;
  size_t n_first = 0;
  std::vector<uint32_t> next(ns.size(), 0);   // the unit's targets dealt so far
  for (int most = 32; most >= WAVE_FEW_LANES; most /= 2) {
    for (uint32_t u = 0; u < ns.size(); ++u) {
      // targets whose chain on half the lanes is too long
      uint32_t end = n_targets;
      if (most > WAVE_FEW_LANES) {
        const uint64_t longest = wave_longest(ns[u], most, limit);
        end = (uint32_t)(std::partition_point(db->h_perm.begin() + next[u], db->h_perm.begin() + n_targets,
                                              [&](uint32_t t) { return db->h_len[t] > longest; }) -
                         db->h_perm.begin());
      }
      const uint32_t first = next[u], count = end - first;
      if (count == 0) continue;
      next[u] = end;
      const int G = wave_lanes(ns[u], most, n_targets / halves * ns.size(), slots);
      segs.push_back({u, first, count, 0, G, NW});
      n_first += most == 32;
    }
  }
  auto items_of = [&](size_t from, size_t to, int warps) {
    uint64_t x = 0;
    for (size_t k = from; k < to; ++k) {
      const uint32_t per = warps * 32 / segs[k].G * halves;
      x += (segs[k].count + per - 1) / per;
    }
    return x;
  };
  // A launch that does not fill the chip, and the longest targets of any, use
  // fewer warps of more CTAs: a chain's step takes 600 cycles on a scheduler of
  // its own and 1,300 beside three others (128 residues against 2,000 targets
  // 0.60 -> 0.54 ms, against 200,000 2.58 -> 2.15).
  int w_all = NW;
  while (w_all > MIN_WARPS && items_of(0, segs.size(), w_all / 2) <= ctas) w_all /= 2;
  int w_first = w_all;
  while (w_first > MIN_WARPS && items_of(0, n_first, w_first / 2) <= ctas / 4) w_first /= 2;
  uint32_t items = 0;
  for (size_t k = 0; k < segs.size(); ++k) {
    segs[k].warps = k < n_first ? w_first : w_all;
    segs[k].item0 = items;
    items += (uint32_t)items_of(k, k + 1, segs[k].warps);
  }
  const unsigned grid = std::min<uint32_t>(items, ctas);

  // Boundary rows: an item takes a row of its longest target per lane group with
  // a target, none if its unit fits one band.  The k-th CTA to start takes its
  // first item in the same step, so never one before item k: its slot holds the
  // largest of the items from there on.  (Slots of every warp by the longest
  // target of all: one query of 2,000 against 100 targets of a million took 3.2
  // GB, now 0.4.)
  auto boundary = [&](const Segment& s, uint32_t tile) -> uint64_t {
    if (ns[s.unit] <= (uint32_t)s.G) return 0;
    const uint32_t per = s.warps * 32 / s.G * halves, at = tile * per;
    return (uint64_t)((std::min(per, s.count - at) + halves - 1) / halves) *
           boundary_row(db->h_len[db->h_perm[s.first + at]]);
  };
  std::vector<uint64_t> slot(grid, 0);
  uint64_t largest = 0;
  for (uint32_t k = (uint32_t)segs.size(), end = items; k-- > 0; end = segs[k].item0) {
    const Segment& s = segs[k];   // needs fall along a segment
    if (end > grid) largest = std::max(largest, boundary(s, std::max(s.item0, grid) - s.item0));
    for (uint32_t x = std::min(end, grid); x-- > s.item0;) slot[x] = largest = std::max(largest, boundary(s, x - s.item0));
  }
  uint64_t b_scr = 0;
  for (uint64_t& s : slot) {
    const uint64_t cells = s;
    s = b_scr;
    b_scr += cells;
  }
  b_scr *= sizeof(uint2);

  WaveArgs W{};
  W.tcodes = db->d_codes; W.toff = db->d_off; W.tlen = db->d_len; W.perm = db->d_perm;
  W.qlen = qs->d_len;
  W.A = A; W.o = o; W.e = e; W.mode = mode; W.fe = fe;
  W.bias = sum_bias(local, o, e, smin);
  W.T = 32767 - std::max(0, smax);
  ProfArgs P{};
  P.qcodes = qs->d_codes; P.qoff = qs->d_off; P.qlen = qs->d_len;
  P.n_strips = (uint32_t)meta.size();
  P.S = d_matrix; P.P = d_pssm;
  P.A = A; P.R = rows; P.form = form;
  W.K = dual ? wave_dual_K(local, o, e, smin) : 0;
  P.dual = dual;
  P.add = (form == LOCAL_SUM ? o + e : form == LOCAL_WRAP ? o : 2 * e) + W.K;
  P.none = dual ? 0 : form == LOCAL_WRAP ? NEG16 : -128;
  if (!local) {
    const bool sg = mode == DSA_SEMIGLOBAL;
    P.pad_row = sg && (fe & DSA_FREE_T_BEGIN) ? P.add : P.add - o;
    P.pad_col = sg && (fe & DSA_FREE_Q_BEGIN) ? P.add : P.add - o;
  }
  const int pw = local ? P.none : P.pad_row;
  W.pad_word = dual ? (uint32_t)pw * 0x01010101u : form == LOCAL_WRAP ? (uint32_t)(pw & 0xFFFF) * 0x10001u : ((uint32_t)pw << 16) + (uint32_t)pw;

  // one upload: segments, strip records, each unit's first strip and strip
  // count, the CTAs' slots
  const size_t b_seg = (segs.size() * sizeof(Segment) + 15) & ~(size_t)15;
  const size_t b_meta = (meta.size() * sizeof(StripMeta) + 15) & ~(size_t)15;
  const size_t b_u = (ns.size() * 4 + 15) & ~(size_t)15;
  const size_t b_slot = (grid * 8 + 15) & ~(size_t)15;
  std::vector<uint8_t> host(b_seg + b_meta + 2 * b_u + b_slot);
  memcpy(host.data(), segs.data(), segs.size() * sizeof(Segment));
  memcpy(host.data() + b_seg, meta.data(), meta.size() * sizeof(StripMeta));
  memcpy(host.data() + b_seg + b_meta, sbase.data(), sbase.size() * 4);
  memcpy(host.data() + b_seg + b_meta + b_u, ns.data(), ns.size() * 4);
  memcpy(host.data() + b_seg + b_meta + 2 * b_u, slot.data(), grid * 8);
  const size_t b_prof = ((size_t)P.n_strips * (A + 1) * rows * (dual ? 1 : 4) + 15) & ~(size_t)15;
  void* buf = nullptr;
  const size_t at_scr = (host.size() + b_prof + 127) & ~(size_t)127;
  const size_t b_all = at_scr + b_scr + 16;
  DSA_TRY(ctx->alloc(&buf, b_all, stream));
  uint8_t* d = static_cast<uint8_t*>(buf);
  cudaError_t err = cudaMemcpyAsync(d, host.data(), host.size(), cudaMemcpyHostToDevice, stream);
  W.segs = reinterpret_cast<const Segment*>(d);
  W.meta = P.meta = reinterpret_cast<const StripMeta*>(d + b_seg);
  W.sbase = reinterpret_cast<const uint32_t*>(d + b_seg + b_meta);
  W.nstrips = reinterpret_cast<const uint32_t*>(d + b_seg + b_meta + b_u);
  W.prof = P.prof = reinterpret_cast<uint32_t*>(d + host.size());
  W.scratch = reinterpret_cast<uint2*>(d + at_scr);
  W.slot = reinterpret_cast<const uint64_t*>(d + b_seg + b_meta + 2 * b_u);
  W.n_segs = (uint32_t)segs.size();
  W.n_items = items;
  W.counter = reinterpret_cast<unsigned long long*>(ctx->d_counters + 4);
  W.out = out;
  W.n_out_t = db->n;
  if (err == cudaSuccess) err = cudaMemsetAsync(W.counter, 0, sizeof(*W.counter), stream);
  if (err == cudaSuccess) {
    const uint64_t words = (uint64_t)P.n_strips * (A + 1) * rows;
    k_wave_profile<<<(unsigned)std::min<uint64_t>((words + 255) / 256, (uint64_t)ctx->sm_count * 8), 256, 0,
                     stream>>>(P);
    kern<<<grid, NT, smem, stream>>>(W);
    ctx->launches += 2;
    err = cudaGetLastError();
  }
  ctx->release(buf, b_all, stream);
  if (err != cudaSuccess) {
    set_error("k_wave launch: %s", cudaGetErrorString(err));
    return DSA_ERR_CUDA;
  }
  return DSA_OK;
}

}  // namespace dsa
