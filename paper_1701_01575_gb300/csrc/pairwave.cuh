// Explicit pairs as small wavefronts, packed int16x2: a group of G lanes (2
// to 32, a power of two) aligns one pair (Sec. II.B.1; any of the three
// algorithms of Sec. II.C.2).  Shared by the planned kernel (k_pairwave.cu)
// and the allocation-free entry point (k_noalloc.cu).
//
// Layout.  The query's rows are cut into blocks of R rows; lane k of the group
// owns blocks 2k (low 16-bit halves) and 2k + 1 (high halves).  At step s the
// low half works on target column s - 2k and the high half on the column
// before it, so a block's top row is the bottom row that the block above
// computed one step earlier: one shuffle each for H and F, joined with the
// lane's own low half by a byte permute.  A pair therefore keeps G lanes busy
// from its first column on, where one thread per pair leaves most of the chip
// idle unless there are hundreds of thousands of pairs, and takes as long as
// its longest pair.  2 G R rows make a band; further bands are chained through
// one boundary row.
//
// Substitution scores come from a profile of the lane's own 2R rows in shared
// memory, a byte per (residue, row): two loads per step give all rows of both
// blocks (the halves are on different columns, so on different residues), and
// one byte permute per packed cell joins and sign-extends them.  Planes of 16
// bytes per lane keep a quarter-warp's loads in different banks whatever
// residues they hold.  No lane reads another lane's profile.
//
// Anchoring.  The query is shifted down by (R - m mod R) mod R padding rows,
// so that row m is the last row of one block; padding rows reproduce row 0.
// Columns before the window (lanes start one after another) and past its end
// hold the padding residue: before the window a block's column-0 state is a
// fixed point of the update with it, so no step needs a bounds test.
//
// Cell update, local (offset binary, Ho = H - o, as in the inter-sequence
// kernel):  E = max(E - e, Ho_left);  t = max(Ho_diag + (S + o), E);
//   H = max(t, F, 0);  Ho = H - o;  F' = max(F - e, Ho).
// Local, summed, where S + o + e >= 0 and no value can pass 16 bits: e j is added
// to the values of column j, which frees E's maximum for the floor:
//   H = max(Ho_diag + (S + o + e), E, F);  Ho = H - o;  F' = max(F - e, Ho);
//   E' = max(E, Ho + e, floor of the next column).
// Cell update, global and semi-global: every value is kept with e (i + j)
// added, so extending a gap adds nothing, and E and F of the next cell are one
// operation each; with G = value + e (i + j) and P = S + 2e + K >= 0:
//   x = G_diag + P - K;  G = max(x, E, F);
//   E' = max(G + (e - o), E);  F' = max(G + (e - o), F)
// The sum is one 32-bit addition of three terms: no half leaves [0, 2^16), so
// nothing carries from one into the other.  Three of the five operations are
// maxima on the half-rate pipe.  (Taking K off after the maxima instead put a
// third operation per row on F's chain: 20,000 protein pairs of 1,024 x 1,024,
// two warps per scheduler, 4.59 ms so and 3.93 now.)
//
// Range.  Local: the saturation rule of the other packed kernels (a best above
// 32767 - max S is rerun in int32 by the caller).  Global and semi-global:
// values with e (i + j) added lie between -3o (less e for each column a lane
// starts before the window) and max(S, 0) min(m, n) + e (m + n + margin);
// pair_wave_range_ok() admits only pairs whose values fit 16 bits, so nothing
// is ever rerun.
#pragma once
#include "dsa_internal.cuh"
#include "dpx.cuh"

#include <type_traits>

namespace dsa {

constexpr int WAVE_WARPS = 4;             // warps per CTA, each on its own
constexpr int WAVE_SM_PITCH = 36;         // bytes per row of the score table (spreads the banks)
constexpr int WAVE_PLANE = 32 * 16;       // profile bytes per residue and half (16 rows)
constexpr int WAVE_PLANE4 = 32 * 4;       // and of the four rows past 16
constexpr int WAVE_WIDE_ALPHABET = 8;     // alphabets whose blocks may have 20 rows
__host__ __device__ constexpr int wave_residue(int R) { return 2 * (WAVE_PLANE + (R > 16 ? WAVE_PLANE4 : 0)); }

// The three forms of the cell update.
enum WaveForm { WAVE_GLOBAL = 0, WAVE_LOCAL = 1, WAVE_LOCAL_SUM = 2 };

struct WaveParams {
  int A, o, e, mode;
  uint32_t fe;
  int K, bias;      // summed forms: see above
};

// K of the global / semi-global update: every table byte is at least 0.
__host__ __device__ inline int pair_wave_K(int o, int e, int smin) {
  int k = -(smin + 2 * e);
  if (o - 2 * e > k) k = o - 2 * e;
  return k > 0 ? k : 0;
}
// The stored value of 0 at cell (0, 0): values fall by 3o below the boundary's
// and by e for each of the up to 63 columns a lane starts before the window.
__host__ __device__ inline int pair_wave_bias(int o, int e, int K) { return 4 * o + 64 * e + K + 64; }
// The byte tables hold every score of this scoring.
__host__ __device__ inline bool pair_wave_tables_ok(bool local, int o, int e, int smax, int smin) {
  if (local) return o >= 1 && o + smax <= 127 && o + smin >= -128;
  const int K = pair_wave_K(o, e, smin);
  return (smax > 0 ? smax : 0) + 2 * e + K <= 127;
}
// Local: the summed form holds this scoring and pairs of up to m x n.
__host__ __device__ inline bool pair_wave_local_sum_ok(int64_t m, int64_t n, int o, int e, int smax,
                                                       int smin) {
  const int64_t up = (int64_t)(smax > 0 ? smax : 0) * (m < n ? m : n) + (int64_t)e * (n + 128);
  return smin + o + e >= 0 && smax + o + e <= 127 && up + 1024 + 4 * o + 64 * e < 65536;
}
// A pair of m x n fits the packed global / semi-global range.
__host__ __device__ inline bool pair_wave_range_ok(int64_t m, int64_t n, int o, int e, int smax,
                                                   int smin) {
  const int K = pair_wave_K(o, e, smin);
  const int64_t up = (int64_t)(smax > 0 ? smax : 0) * (m < n ? m : n) + (int64_t)e * (m + n + 256);
  return up + pair_wave_bias(o, e, K) + 512 < 65536;
}

// Shared-memory bytes of a CTA: the score table, then per warp the profile
// and (local) the parked columns.
__host__ __device__ inline uint32_t pair_wave_table_bytes(int A) {
  return ((uint32_t)(A + 2) * WAVE_SM_PITCH + 127u) / 128u * 128u;
}
__host__ __device__ inline uint32_t pair_wave_warp_bytes(int A, bool local) {
  const int R = A <= WAVE_WIDE_ALPHABET ? 20 : 16;
  return (uint32_t)(A + 1) * wave_residue(R) + (local ? 2u * R * 32u * 2u : 0u);
}
// of a CTA's warps, and the most any alphabet takes
__host__ __device__ inline uint32_t pair_wave_smem(int A, bool local) {
  return pair_wave_table_bytes(A) + (uint32_t)WAVE_WARPS * pair_wave_warp_bytes(A, local);
}
// offset of the parked columns behind the profile
__host__ __device__ inline uint32_t pair_wave_park_offset(int A) {
  return (uint32_t)(A + 1) * wave_residue(A <= WAVE_WIDE_ALPHABET ? 20 : 16);
}

#ifdef __CUDACC__

// Score table rows by query residue (row A: padding rows above the query, row
// A + 1: rows below it), bytes by target residue (entry A: the padding
// residue).  S(q, a) is the caller's matrix.
template <int FORM, class Fn>
__device__ __forceinline__ void pair_wave_table(const WaveParams& W, uint8_t* tab, Fn S) {
  const bool sg = W.mode == DSA_SEMIGLOBAL;
  const bool qb = sg && (W.fe & DSA_FREE_Q_BEGIN), tb = sg && (W.fe & DSA_FREE_T_BEGIN);
  const int z = 2 * W.e + W.K;   // S = 0
  for (int x = threadIdx.x; x < (W.A + 2) * (WAVE_SM_PITCH); x += blockDim.x) {
    const int q = x / WAVE_SM_PITCH, a = x % WAVE_SM_PITCH;
    constexpr bool LOCAL = FORM != WAVE_GLOBAL;
    int v = FORM == WAVE_LOCAL ? -128 : 0;   // below any score
    if (q < W.A && a < W.A)
      v = S(q, a) + (FORM == WAVE_LOCAL_SUM ? W.o + W.e : LOCAL ? W.o : z);
    else if (!LOCAL && q < W.A && a == W.A) v = qb ? z : z - W.o;
    else if (!LOCAL && q == W.A) v = (a == W.A || tb) ? z : z - W.o;
    tab[x] = (uint8_t)(int8_t)v;
  }
}

// One warp, 32 / G pairs (group g = lane / G; m = n = 0: no pair).  q, t, m, n,
// scr (the group's boundary row, for queries of more than one band) and the
// outputs are the group's; the result is valid on the group's first lane:
// local: score and 1-based end cell (0 when nothing scores); others: score and
// end cell (i, j) with i in 0..m, j in 0..n.
template <int FORM, int R>
__device__ __forceinline__ void pair_wave_run(const WaveParams& W, const uint8_t* tab, uint8_t* prof,
                                              uint2* park, int G, const uint8_t* q,
                                              const uint8_t* t, int m, int n, uint32_t* scr,
                                              int& out_s, int& out_i, int& out_j) {
  static_assert(R % 4 == 0 && R <= 20, "rows per block");
  constexpr bool LOCAL = FORM != WAVE_GLOBAL, LSUM = FORM == WAVE_LOCAL_SUM;
  constexpr int RES = wave_residue(R), Q = R / 4;
  constexpr unsigned FULL = 0xFFFFFFFFu;
  constexpr uint32_t BIAS2 = 0x80008000u;
  const int lane = threadIdx.x & 31, k = lane & (G - 1);
  const int o = W.o, e = W.e, A = W.A;
  const bool sg = W.mode == DSA_SEMIGLOBAL;
  const bool qb_free = sg && (W.fe & DSA_FREE_Q_BEGIN), qe_free = sg && (W.fe & DSA_FREE_Q_END);
  const bool tb_free = sg && (W.fe & DSA_FREE_T_BEGIN), te_free = sg && (W.fe & DSA_FREE_T_END);
  const uint32_t neg_e2 = pack2(-e, -e), o2 = pack2(o, 0) + ((uint32_t)o << 16);
  const uint32_t K2 = (uint32_t)W.K * 0x10001u;
  const uint32_t c2 = pack2(e - o, e - o);
  const uint32_t e2 = (uint32_t)e * 0x10001u;
  const int jl0 = -2 * k;   // the low half's column before step 1
  // local: H = 0 as H - o (summed: at the halves' columns before step 1)
  const uint32_t mo2 = LSUM ? pack2(W.bias + e * jl0 - o, W.bias + e * (jl0 - 1) - o) : pack2(-o, -o) ^ BIAS2;
  const int pad = (R - m % R) % R, mp = m + pad;
  const int band = 2 * G * R;
  const int nb = (mp + band - 1) / band;
  int nbmax = nb, nmax = n, nmin = n;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    nbmax = max(nbmax, __shfl_xor_sync(FULL, nbmax, s));
    nmax = max(nmax, __shfl_xor_sync(FULL, nmax, s));
    nmin = min(nmin, __shfl_xor_sync(FULL, nmin, s));
  }
  // value of H at column 0, row i' (padded rows, 1-based; row 0 and padding
  // rows: 0), and of F entering row i' + 1 there, with e (i' + j) added
  auto hv = [&](int i, int j) {
    const int h = (i <= pad || qb_free) ? 0 : -(o + (i - pad - 1) * e);
    return W.bias + h + e * (i + j);
  };
  auto fv = [&](int i, int j) {
    const int f = (i <= pad || qb_free) ? -o : -(o + (i - pad) * e);
    return W.bias + f + e * (i + 1 + j);
  };
  auto row0 = [&](int j) { return (j == 0 || tb_free) ? 0 : -(o + (j - 1) * e); };

  // local: running best per half.  others: column n's best (free query end),
  // H[m][n] and row m's best column, held by the lane that has them
  int best_lo = 0, best_hi = 0, bj_lo = 0, bj_hi = 0, bi_lo = 0, bi_hi = 0, gbest = 0;
  int cb = qe_free ? row0(n) : INT32_MIN, ci = 0, hmn = INT32_MIN, rj = 0;
  int rbest = INT32_MIN;
  uint8_t* const plo = prof + lane * 16;
  park += lane;   // parked columns: [half][4 rows of 16 bits][lane]

  for (int b = 0; b < nbmax; ++b) {
    const int base = b * band + 2 * k * R;   // rows above the low block
    // ---- the lane's profile ----
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const uint32_t* row[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = base + x * R + r - pad;   // 0-based query row
        const int c = i < 0 ? A : (i < m ? (int)q[i] : A + 1);
        row[r] = reinterpret_cast<const uint32_t*>(tab + c * WAVE_SM_PITCH);
      }
      for (int a = 0; a <= A; a += 4) {
        uint32_t w[4][Q < 4 ? 4 : Q];
#pragma unroll
        for (int g = 0; g < R / 4; ++g) {   // 4 rows x 4 residues, transposed
          const uint32_t w0 = row[4 * g][a / 4], w1 = row[4 * g + 1][a / 4];
          const uint32_t w2 = row[4 * g + 2][a / 4], w3 = row[4 * g + 3][a / 4];
          const uint32_t p0 = prmt(w0, w1, 0x5140), p1 = prmt(w0, w1, 0x7362);
          const uint32_t p2 = prmt(w2, w3, 0x5140), p3 = prmt(w2, w3, 0x7362);
          w[0][g] = prmt(p0, p2, 0x5410);
          w[1][g] = prmt(p0, p2, 0x7632);
          w[2][g] = prmt(p1, p3, 0x5410);
          w[3][g] = prmt(p1, p3, 0x7632);
        }
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (a + y <= A) {
            uint8_t* dst = plo + (a + y) * RES + x * WAVE_PLANE;
            if (R == 8)
              *reinterpret_cast<uint2*>(dst) = make_uint2(w[y][0], w[y][1]);
            else
              *reinterpret_cast<uint4*>(dst) =
                  make_uint4(w[y][0], w[y][1], w[y][2], R >= 16 ? w[y][3] : 0u);
            if (R > 16)
              *reinterpret_cast<uint32_t*>(prof + (a + y) * RES + 2 * WAVE_PLANE + x * WAVE_PLANE4 +
                                           lane * 4) = w[y][Q - 1];
          }
      }
    }
    // ---- column-0 state ----
    uint32_t Ho[R], E[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (LOCAL) {
        Ho[r] = mo2;
        E[r] = LSUM ? mo2 + o2 + e2 : pack2(NEG16, NEG16) ^ BIAS2;
      } else {
        Ho[r] = pack2(hv(base + r + 1, jl0), hv(base + R + r + 1, jl0 - 1));
        E[r] = add2(Ho[r], c2);   // E of column 1 opens from column 0
      }
    }
    uint32_t diag = LOCAL ? mo2 : pack2(hv(base, jl0), hv(base + R, jl0 - 1));
    uint32_t sendH = Ho[R - 1];
    uint32_t sendF = LOCAL ? mo2 : pack2(fv(base + R, jl0), fv(base + 2 * R, jl0 - 1));
    // row m's best so far as a threshold that moves with e j (a half that does
    // not hold row m: never passed); the candidate (m, 0) starts it
    uint32_t rthr = 0xFFFFFFFFu, rinc = 0;
    const bool own_lo = !LOCAL && m > 0 && base + R == mp;
    const bool own_hi = !LOCAL && m > 0 && base + 2 * R == mp;
    if (te_free && own_lo) { rthr = 0xFFFF0000u | (uint32_t)hv(mp, jl0); rinc = (uint32_t)e; }
    if (te_free && own_hi) { rthr = 0x0000FFFFu | (uint32_t)hv(mp, jl0 - 1) << 16; rinc = (uint32_t)e << 16; }
    // columns whose maximum reaches the best of their half, or the best that
    // the group's lanes had at the last exchange, trigger
    uint32_t thr2 = 0xFFFFFFFFu;
    uint32_t flo2 = mo2;   // summed: H = 0 as H - o at the halves' columns
    auto set_thr = [&]() {
      if (LOCAL && b < nb)
        thr2 = pack2(max(max(best_lo, gbest) - 1, 0), max(max(best_hi, gbest) - 1, 0)) +
               (LSUM ? flo2 + o2 : BIAS2);
    };
    set_thr();
    int pend = 0;
    const bool keep = b + 1 < nb && k == G - 1;   // this band's bottom row is read again
    // lane 0's input row in the high halves (the low halves of the lane above
    // are its own high ones): row 0 at column j, or the band above
    uint32_t inH = mo2 << 16, inF = mo2 << 16, inc = LSUM ? (uint32_t)e << 16 : 0u, inw = 0;
    if (!LOCAL) {
      // row 0: constant from column 1 on, or rising by e with a free begin
      const uint32_t v = (uint32_t)(W.bias + (tb_free ? 0 : e - o));
      inH = v << 16;
      inF = (v + (uint32_t)(e - o)) << 16;
      inc = tb_free ? (uint32_t)e << 16 : 0u;
    }
    if (b > 0 && k == 0 && n > 0) inw = scr[0];
    uint32_t a_hi = (uint32_t)A * RES;   // the residue of the high half's column, as a profile offset

    // one step: the low half's column j, the high half's j - 1, with the low
    // half's residue (as an offset); EDGE: some lane may be before its window's
    // start or at its end
    int j = jl0;
    auto step = [&](uint32_t a_lo, int s, auto edge_c) {
      constexpr bool EDGE = decltype(edge_c)::value;
      ++j;
      uint32_t upH = __shfl_up_sync(FULL, sendH, 1);
      uint32_t upF = __shfl_up_sync(FULL, sendF, 1);
      if (b > 0) {
        inH = inw << 16;
        inF = inw & 0xFFFF0000u;
        if (k == 0 && s < n) inw = scr[s];
      } else if (FORM != WAVE_LOCAL) {
        inH += inc;
        inF += inc;
      }
      uint32_t fln2 = 0;   // summed local: the floor of the next column
      if (LSUM) {
        flo2 += e2;
        if (b < nb) thr2 += e2;
        fln2 = flo2 + o2 + e2;
      }
      upH = k == 0 ? inH : upH;
      upF = k == 0 ? inF : upF;
      const uint32_t topH = prmt(upH, sendH, 0x5432);
      uint32_t F = prmt(upF, sendF, 0x5432);
      uint32_t pl[Q < 4 ? 4 : Q], ph[Q < 4 ? 4 : Q];
      if (R == 8) {
        const uint2 v = *reinterpret_cast<const uint2*>(plo + a_lo);
        const uint2 u = *reinterpret_cast<const uint2*>(plo + WAVE_PLANE + a_hi);
        pl[0] = v.x; pl[1] = v.y; ph[0] = u.x; ph[1] = u.y;
      } else {
        const uint4 v = *reinterpret_cast<const uint4*>(plo + a_lo);
        const uint4 u = *reinterpret_cast<const uint4*>(plo + WAVE_PLANE + a_hi);
        pl[0] = v.x; pl[1] = v.y; pl[2] = v.z; pl[3] = v.w;
        ph[0] = u.x; ph[1] = u.y; ph[2] = u.z; ph[3] = u.w;
        if (R > 16) {
          pl[Q - 1] = *reinterpret_cast<const uint32_t*>(prof + 2 * WAVE_PLANE + lane * 4 + a_lo);
          ph[Q - 1] = *reinterpret_cast<const uint32_t*>(prof + 2 * WAVE_PLANE + WAVE_PLANE4 + lane * 4 + a_hi);
        }
      }
      a_hi = a_lo;
      uint32_t d = diag;
      diag = topH;
      uint32_t cm = LSUM ? 0u : BIAS2, hprev = cm;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const uint32_t bsel = r & 3;
        const uint32_t sp = prmt(pl[r / 4], ph[r / 4],
                                 bsel | (8 + bsel) << 4 | (4 + bsel) << 8 | (12 + bsel) << 12);
        const uint32_t old = Ho[r];
        if (LSUM) {
          const uint32_t h = max3_2u(d + sp, E[r], F);
          const uint32_t ho = h - o2;
          F = addmax2u(F, neg_e2, ho);
          E[r] = max3_2u(E[r], ho + e2, fln2);
          Ho[r] = ho;
          if (r & 1) cm = max3_2u(cm, hprev, h);
          else hprev = h;
        } else if (LOCAL) {
          E[r] = addmax2u(E[r], neg_e2, old);
          const uint32_t x = addmax2u(d, sp, E[r]);
          const uint32_t h = max3_2u(x, F, BIAS2);
          Ho[r] = h - o2;
          F = addmax2u(F, neg_e2, Ho[r]);
          if (r & 1) cm = max3_2u(cm, hprev, h);
          else hprev = h;
        } else {
          const uint32_t h = max3_2u(d + sp - K2, E[r], F);
          Ho[r] = h;
          E[r] = addmax2u(h, c2, E[r]);
          F = addmax2u(h, c2, F);
        }
        d = old;
      }
      sendH = Ho[R - 1];
      sendF = F;
      if (b + 1 < nbmax && keep && (uint32_t)(j - 2) < (uint32_t)n) scr[j - 2] = prmt(sendH, sendF, 0x7632);
      if (LOCAL) {
        if (__vmaxu2(cm, thr2) != thr2) {
          const int cl = (int)(cm & 0xFFFFu) - (LSUM ? (int)(flo2 & 0xFFFFu) + o : 0x8000);
          const int ch = (int)(cm >> 16) - (LSUM ? (int)(flo2 >> 16) + o : 0x8000);
          const bool lo = cl >= gbest && cl > best_lo - (j < bj_lo ? 1 : 0);
          const bool hi = ch >= gbest && ch > best_hi - (j - 1 < bj_hi ? 1 : 0);
          // lanes that raise either half park it in one pass
          if (lo | hi) {
            auto keep_half = [&](uint2* p, uint32_t sel) {
#pragma unroll
              for (int r = 0; r < R; r += 4)
                p[r / 4 * 32] = make_uint2(prmt(Ho[r], Ho[r + 1], sel), prmt(Ho[r + 2], Ho[r + 3], sel));
            };
            keep_half(park + (lo ? 0 : Q * 32), lo ? 0x5410u : 0x7632u);
            if (lo & hi) keep_half(park + Q * 32, 0x7632u);
            if (lo) { best_lo = cl; bj_lo = j; pend |= 1; }
            if (hi) { best_hi = ch; bj_hi = j - 1; pend |= 2; }
          }
          set_thr();
        }
      } else {
        if (te_free) {
          rthr += rinc;
          if (__vmaxu2(sendH, rthr) != rthr) {
            const int jj = own_lo ? j : j - 1;
            if (jj >= 1 && jj <= n) {
              rthr = own_lo ? (rthr & 0xFFFF0000u) | (sendH & 0xFFFFu)
                            : (rthr & 0x0000FFFFu) | (sendH & 0xFFFF0000u);
              rj = jj;
              rbest = (int)(own_lo ? sendH & 0xFFFFu : sendH >> 16) - W.bias - e * (mp + jj);
            }
          }
        }
        if (EDGE && (uint32_t)(j - n) <= 1u) {   // column n, low half then high half
          const int x = j - n, sh = 16 * x;
          if (x ? own_hi : own_lo)
            hmn = (int)((sendH >> sh) & 0xFFFFu) - W.bias - e * (mp + n);
          if (qe_free) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int i = base + x * R + r + 1;
              const int v = (int)((Ho[r] >> sh) & 0xFFFFu) - W.bias - e * (i + n);
              if (i > pad && i <= mp && v > cb) { cb = v; ci = i - pad; }
            }
          }
        }
      }
    };
    // Blocks of 4 steps, their residues loaded a block ahead: inside every
    // window two aligned words (never past the window) for a funnel shift, at
    // its ends four bytes with the padding residue outside it.
    const int steps = nmax + 2 * G - 1;
    auto inside = [&](int s0) { return s0 >= 2 * G + 2 && s0 + 8 <= nmin; };
    const uint32_t sh = 8u * (uint32_t)((uintptr_t)(t - 2 * k) & 3);
    auto words = [&](int s0) -> uint2 {
      if (!inside(s0)) {
        uint32_t w = 0;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int x = s0 - 2 * k + y;
          w |= ((uint32_t)x < (uint32_t)n ? (uint32_t)t[x] : (uint32_t)A) << (8 * y);
        }
        return make_uint2(w, 0);
      }
      const uint32_t* p = reinterpret_cast<const uint32_t*>((uintptr_t)(t + (s0 - 2 * k)) & ~(uintptr_t)3);
      return make_uint2(p[0], p[1]);
    };
    uint2 nxt = words(0);
    for (int s0 = 0; s0 < steps; s0 += 4) {
      if (LOCAL && (s0 & 31) == 28) {
        int v = max(best_lo, best_hi);
        for (int w = G / 2; w > 0; w >>= 1) v = max(v, __shfl_xor_sync(FULL, v, w));
        gbest = v;
        set_thr();
      }
      const uint2 cur = nxt;
      nxt = words(s0 + 4);
      if (inside(s0)) {
        const uint32_t r4 = __funnelshift_r(cur.x, cur.y, sh);
#pragma unroll
        for (int y = 0; y < 4; ++y) step(((r4 >> (8 * y)) & 0xFFu) * RES, s0 + 1 + y, std::false_type{});
      } else {
#pragma unroll 1
        for (int y = 0; y < 4; ++y) step(((cur.x >> (8 * y)) & 0xFFu) * RES, s0 + 1 + y, std::true_type{});
      }
    }
    if (!LOCAL && te_free && (own_lo || own_hi) && rj == 0)
      rbest = qb_free ? 0 : -(o + (m - 1) * e);   // (m, 0) was never passed
    if (LOCAL) {   // rows of the parked columns
      auto row = [&](int x, int best, int bj) {   // first row of half x holding the maximum
        const uint16_t want = (uint16_t)(best - o + (LSUM ? W.bias + e * bj : 0x8000));
        int rr = 0;
        for (int r = R - 1; r >= 0; --r)
          if (reinterpret_cast<const uint16_t*>(park + (x * Q + r / 4) * 32)[r & 3] == want) rr = r;
        return base + x * R + rr + 1 - pad;
      };
      if (pend & 1) bi_lo = row(0, best_lo, bj_lo);
      if (pend & 2) bi_hi = row(1, best_hi, bj_hi);
    }
    __syncwarp();
  }
  if (LOCAL) {
    if (best_hi > best_lo || (best_hi == best_lo && best_hi > 0 &&
                              (bj_hi < bj_lo || (bj_hi == bj_lo && bi_hi < bi_lo)))) {
      best_lo = best_hi; bj_lo = bj_hi; bi_lo = bi_hi;
    }
    for (int w = G / 2; w > 0; w >>= 1) {
      const int s2 = __shfl_xor_sync(FULL, best_lo, w);
      const int j2 = __shfl_xor_sync(FULL, bj_lo, w);
      const int i2 = __shfl_xor_sync(FULL, bi_lo, w);
      if (s2 > best_lo || (s2 == best_lo && s2 > 0 && (j2 < bj_lo || (j2 == bj_lo && i2 < bi_lo)))) {
        best_lo = s2; bj_lo = j2; bi_lo = i2;
      }
    }
    out_s = best_lo;
    out_i = best_lo > 0 ? bi_lo : 0;
    out_j = best_lo > 0 ? bj_lo : 0;
  } else {
    for (int w = G / 2; w > 0; w >>= 1) {
      const int s2 = __shfl_xor_sync(FULL, cb, w), i2 = __shfl_xor_sync(FULL, ci, w);
      if (s2 > cb || (s2 == cb && i2 < ci)) { cb = s2; ci = i2; }
      // one lane holds row m
      hmn = max(hmn, __shfl_xor_sync(FULL, hmn, w));
      const int r2 = __shfl_xor_sync(FULL, rbest, w), rj2 = __shfl_xor_sync(FULL, rj, w);
      if (r2 > rbest) { rbest = r2; rj = rj2; }
    }
    int bs = hmn, bi = m, bj = n;   // (m, n); then column n, then row m
    if (qe_free && (cb > bs || (cb == bs && ci < bi))) { bs = cb; bi = ci; }
    if (te_free && (rbest > bs || (rbest == bs && rj < bj))) { bs = rbest; bi = m; bj = rj; }
    out_s = bs;
    out_i = bi;
    out_j = bj;
  }
}

#endif  // __CUDACC__

}  // namespace dsa
