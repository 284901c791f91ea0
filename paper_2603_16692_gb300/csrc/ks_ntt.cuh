// Negacyclic NTT stages on a shared-memory tile (device side), with the tile
// geometry fixed at compile time.
//
// Transform (ring x^N + 1): forward Cooley-Tukey stages s = 0..logN-1 with
// m = 2^s, t = N/2^(s+1) and twiddle psi^brv(m+i) for block i; this gives slot
// k = a(psi^(2 brv(k)+1)) (bit-reversed evaluation order). The inverse runs the
// Gentleman-Sande stages in reverse with psi^-brv(m+i), then scales by N^-1.
//
// The inverse twiddle of block i at stage s is psi^-brv(2^s + i) = -psi^brv(2^s + i'),
// with i' = i XOR (2^s - 1) (psi^N = -1, and brv maps the complement of i to N minus
// the exponent). The inverse row pass therefore reads the forward row table: the slab
// of the mirrored row tile, mirrored inside (row g -> G-1-g, block c -> 2^ls-1-c),
// and its Gentleman-Sande butterflies take (Y - X) w instead of (X - Y)(-w).
//
// N = N1 * N2. The column pass runs stages 0..log N1-1 on the N2 columns (each an
// N1-point transform with twiddle index 2^ls + c for local stage ls, block c);
// the row pass runs the remaining stages on the N1 rows of N2 contiguous points
// (twiddle index (N1 + row) 2^ls + c). For N <= 2048 one row pass does all.
//
// A tile holds G = 2^LOGG sub-transforms of M = 2^LOGM points; point x of
// sub-transform g lives at s[x*P + g] (P = G+1 for G > 1: an odd pitch keeps
// 64-bit accesses free of bank conflicts). Twiddles sit in shared memory:
// column pass: tw[k], k = 2^ls + c (the first N1 entries of the table);
// row pass: tw[g * M + row_tw(ls, c)] (the tile's rows one after another; see row_tw).
//
// Each round moves 2^R points of one butterfly group into registers, runs R
// stages there (radix-2^R), and writes them back; every offset is a constant.
#pragma once
#include "ks_arith.cuh"
#include "ks_internal.h"

namespace ks {

// Compile-time geometry of the two passes for N = 2^LOGN (also used on the host
// to lay out the row-pass twiddle table by row tile).
__host__ __device__ constexpr int geo_loga(int logn) { return logn <= 11 ? 0 : logn / 2; }
// Tiles of the shared-memory rounds (the persistent batch; one tile per limb at the
// single-pass sizes). Column pass: 2^10 points up to N = 2^15, 2^11 above. Row pass: 2^9
// points up to N = 2^15, 2^10 above.
__host__ __device__ constexpr int geo_tile_log_col(int logn) {
  return logn <= 11 ? logn : (logn >= 16 ? 11 : 10);
}
__host__ __device__ constexpr int geo_tile_log_row(int logn) {
  return logn <= 11 ? logn : (logn <= 15 ? 9 : 10);
}

// Entry of (local stage ls, block c) in a row's twiddle slab of the two-pass sizes: the
// first kRowHead stages stage-major, then, for the 2^kRowHead sub-blocks of a row that one
// thread (or a few) finishes in registers, each entry of the sub-block's tree for all the
// sub-blocks side by side: lanes that work on consecutive sub-blocks read consecutive
// 16-byte entries (stage-major they would be 2^(ls - kRowHead) entries apart, an up to
// 8-way bank conflict).
constexpr int kRowHead = 4;
__host__ __device__ constexpr int row_tw(int ls, int c) {
  return ls < kRowHead ? (1 << ls) - 1 + c
                       : (1 << kRowHead) - 1 +
                             (((1 << (ls - kRowHead)) - 1 + (c & ((1 << (ls - kRowHead)) - 1)))
                              << kRowHead) +
                             (c >> (ls - kRowHead));
}

// RL: log2 of the radix of the register rounds; a thread holds 2^RL points.
// ROW: geometry of the row pass (1) or of the column pass (0); a kernel runs one pass
// and uses only that pass's fields.
template <int LOGN, int RL_, int ROW>
struct GeoT {
  static constexpr int RL = RL_;
  static constexpr int LOGA = geo_loga(LOGN);  // log N1
  static constexpr int LOGB = LOGN - LOGA;     // log N2
  static constexpr int TILE_LOG = ROW ? geo_tile_log_row(LOGN) : geo_tile_log_col(LOGN);
  static constexpr int LOGGC = LOGA == 0 ? 0 : TILE_LOG - LOGA;  // columns per column tile
  static constexpr int LOGGR = TILE_LOG - LOGB;                  // rows per row tile
  static constexpr int TILE = 1 << TILE_LOG;
  static constexpr int NT = (TILE >> RL) < 32 ? 32 : (TILE >> RL);  // one group per thread
  static constexpr int EPT = (TILE + NT - 1) / NT;           // tile elements per thread
  static constexpr int GC = 1 << LOGGC, GR = 1 << LOGGR;
  static constexpr int PC = GC == 1 ? 1 : GC + 1;
  static constexpr int PR = GR == 1 ? 1 : GR + 1;
  static constexpr int N1 = 1 << LOGA, N2 = 1 << LOGB;
  static constexpr int TWC = N1;                  // column-pass twiddles per tile
  // row-pass twiddles per tile: two-pass sizes hold N2 entries per row (the last unused)
  static constexpr int TWR = LOGA == 0 ? N2 - 1 : N2 * GR;
  // ... in shared memory: a row's slab one entry longer, so that lanes on several rows of a
  // tile read different banks
  static constexpr int TWS = LOGA == 0 ? TWR : (N2 + 1) * GR;
  static constexpr int SMEM_COL = (N1 * PC) * 8 + TWC * 16;
  static constexpr int SMEM_ROW = (N2 * PR) * 8 + TWS * 16;
};

// Butterflies by class of the modulus (mod_class):
//  fast  (m < 2^51): no reduction of the upper input, approximate Shoup product T in
//        [0, 4m). Forward: each stage raises the bound by 4m, so a column pass (<= 8
//        stages) starting below 2m (or 16m, see mid) ends below 48m and the row pass
//        (<= 9 stages) below kFwdLazy m with a column start below 2m; 11 single-pass
//        stages end below 46m. Inverse: canonical inputs; the k-th processed stage adds
//        without reduction and biases the difference by m 2^(k+1) (>= the bound of both
//        inputs), so after K stages all values are below m 2^(K+1) <= 2^13 m < 2^64.
//  mid   (m < 2^60, the special primes): the same product; four bits of headroom, so the
//        upper input is brought below 8m by one conditional subtraction on every other
//        stage. Forward: even local stages take inputs below 16m (X < 8m after the
//        subtraction, outputs below 12m), odd ones inputs below 12m (outputs below 16m).
//        Inverse: values below 8m, one subtraction of 8m from the sum. Measured: 36 cycles
//        per forward butterfly against 43.8 for the exact form below.
//  exact (m < 2^62): Harvey's butterflies, forward values in [0, 4m), inverse in [0, 2m).
enum { CLS_EXACT = 0, CLS_FAST = 1, CLS_MID = 2 };
__device__ __forceinline__ int mod_class(u64 m) {
  return m < kFastModulus ? CLS_FAST : m < kMidModulus ? CLS_MID : CLS_EXACT;
}

template <int CLS>
__device__ __forceinline__ void bfly_fwd_c(u64 &a, u64 &b, const ulonglong2 w, u64 m, int ls) {
  u64 X = a;
  if (CLS == CLS_EXACT) {
    X = csub(X, 2 * m);
    const u64 T = shoup(b, w.x, w.y, m);
    a = X + T;
    b = X - T + 2 * m;
  } else {
    if (CLS == CLS_MID && (ls & 1) == 0) X = csub(X, 8 * m);
    const u64 T = shoup4(b, w.x, w.y, m);
    a = X + T;
    b = X - T + 4 * m;
  }
}

// bias: m 2^(k + 1) for the k-th processed stage (the fast class's). NEG: the twiddle is
// given negated (mirrored tables).
template <int CLS, bool NEG>
__device__ __forceinline__ void bfly_inv_c(u64 &a, u64 &b, const ulonglong2 w, u64 m, u64 bias) {
  const u64 X = a, Y = b, D = NEG ? Y - X : X - Y;
  const u64 S = X + Y;
  if (CLS == CLS_EXACT) {
    a = csub(S, 2 * m);
    b = shoup(D + 2 * m, w.x, w.y, m);
  } else if (CLS == CLS_MID) {
    a = csub(S, 8 * m);
    b = shoup4(D + 8 * m, w.x, w.y, m);
  } else {
    a = S;
    b = shoup4(D + bias, w.x, w.y, m);
  }
}

// Exact sum of 64 x 64-bit products: value lo + 2^32 mid + 2^64 hi. The middle products
// are summed on their own, so a term takes four 32x32->64 products and three 64-bit adds
// (19 cycles a warp against 28.7 for a carry chain over the whole 128 bits). mid must stay
// below 2^63: the caller folds in time.
struct Mac3 {
  u64 lo, hi, mid;
  __device__ __forceinline__ void add(u64 y, u64 k) {
    const uint32_t yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
    const uint32_t kl = (uint32_t)k, kh = (uint32_t)(k >> 32);
    const u64 l = mul_wide(yl, kl), h = mul_wide(yh, kh);
    mid += mul_wide(yl, kh) + mul_wide(yh, kl);
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(lo), "+l"(hi) : "l"(l), "l"(h));
  }
  __device__ __forceinline__ void fold() {
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;"
        : "+l"(lo), "+l"(hi)
        : "l"(mid << 32), "l"(mid >> 32));
    mid = 0;
  }
  // value * 2^-64 mod m, canonical, for a value below m 2^64 and mid below 2^63: two 32-bit
  // Montgomery steps (inv = m^-1 mod 2^32), each taking off u m with u the low word times
  // inv; six products against nine and about half the instructions of fold() and a 64-bit
  // step.
  __device__ __forceinline__ u64 reduce(u64 m, uint32_t inv) const {
    const uint32_t ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
    const uint32_t u0 = (uint32_t)lo * inv;
    const long long t = (long long)(mid + (lo >> 32) - (mul_wide(u0, ml) >> 32)) -
                        (long long)mul_wide(u0, mh);
    const uint32_t u1 = (uint32_t)t * inv;
    const u64 r = hi + (u64)(t >> 32) - (mul_wide(u1, ml) >> 32) - mul_wide(u1, mh) + m;
    return csub(r, m);
  }
};
// The canonical residue of a sum; exact moduli, whose mid may pass 2^63, by fold() and the
// 64-bit step.
__device__ __forceinline__ u64 mac_reduce(Mac3 &s, const ModInfo &mi, u64 m, uint32_t inv,
                                          int cls) {
  if (cls != CLS_EXACT) return s.reduce(m, inv);
  s.fold();
  return csub(redc(U128{s.lo, s.hi}, m, mi.minv), m);
}

template <int LOGM, int LOGG, int P, int NT, bool ROW, bool INV, int LS0, int R, int CLS>
__device__ __forceinline__ void ntt_round(u64 *s, const ulonglong2 *tw, u64 m) {
  constexpr int SUB = LOGM - LS0 - R;
  constexpr int NG = 1 << (LOGM - R + LOGG);
  const int tid = threadIdx.x;
#pragma unroll
  for (int it = 0; it < (NG + NT - 1) / NT; ++it) {
    const int grp = tid + it * NT;
    if (NG % NT != 0 && grp >= NG) break;
    const int g = grp & ((1 << LOGG) - 1);
    const int rest = grp >> LOGG;
    const int lo = rest & ((1 << SUB) - 1);
    const int hi = rest >> SUB;
    u64 *base = s + ((hi << (LOGM - LS0)) + lo) * P + g;
    u64 v[1 << R];
#pragma unroll
    for (int u = 0; u < (1 << R); ++u) v[u] = base[(u << SUB) * P];
    if (!INV) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int half = 1 << (R - 1 - q);
        // twiddle index of local stage LS0+q, block (hi << q) + (u >> (R-q)); row tiles
        // with several rows (two-pass sizes) take the row-major slab
        const ulonglong2 *twq =
            ROW ? (LOGG ? tw + g * ((1 << LOGM) + 1) : tw + (1 << (LS0 + q)) - 1 + (hi << q))
                : tw + (1 << (LS0 + q)) + (hi << q);
#pragma unroll
        for (int u = 0; u < (1 << R); ++u) {
          if (u & half) continue;
          const ulonglong2 w =
              twq[ROW && LOGG ? row_tw(LS0 + q, (hi << q) + (u >> (R - q))) : (u >> (R - q))];
          bfly_fwd_c<CLS>(v[u], v[u + half], w, m, LS0 + q);
        }
      }
    } else {
#pragma unroll
      for (int q = R - 1; q >= 0; --q) {
        const int half = 1 << (R - 1 - q);
        // row pass: the forward slab of the mirrored tile, row g' = G - 1 - g, block
        // c' = 2^ls - 1 - c (negated twiddles)
        const ulonglong2 *twq =
            ROW ? (LOGG ? tw + ((1 << LOGG) - 1 - g) * ((1 << LOGM) + 1)
                        : tw + (2 << (LS0 + q)) - 2 - (hi << q))
                : tw + (1 << (LS0 + q)) + (hi << q);
        const u64 bias = m << (LOGM - (LS0 + q));
#pragma unroll
        for (int u = 0; u < (1 << R); ++u) {
          if (u & half) continue;
          if (ROW) {
            const int c = (hi << q) + (u >> (R - q));
            const ulonglong2 w =
                LOGG ? twq[row_tw(LS0 + q, (1 << (LS0 + q)) - 1 - c)] : twq[-(u >> (R - q))];
            bfly_inv_c<CLS, true>(v[u], v[u + half], w, m, bias);
          } else {
            const ulonglong2 w = twq[u >> (R - q)];
            bfly_inv_c<CLS, false>(v[u], v[u + half], w, m, bias);
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < (1 << R); ++u) base[(u << SUB) * P] = v[u];
  }
}

// Barrier of BARN threads of the block (the others run another role or another group).
template <int BARN>
__device__ __forceinline__ void round_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(BARN) : "memory");
}

// Forward stages 0..LOGM-1 of every sub-transform in the tile, in rounds of at
// most RM stages (bounds: see the butterflies). Caller syncs before; each round syncs
// after.
template <int LOGM, int LOGG, int P, int NT, bool ROW, int RM, int CLS, int LS0 = 0>
__device__ __forceinline__ void tile_fwd_t(u64 *s, const ulonglong2 *tw, u64 m) {
  if constexpr (LS0 < LOGM) {
    constexpr int R = (LOGM - LS0) >= RM ? RM : (LOGM - LS0);
    ntt_round<LOGM, LOGG, P, NT, ROW, false, LS0, R, CLS>(s, tw, m);
    __syncthreads();
    tile_fwd_t<LOGM, LOGG, P, NT, ROW, RM, CLS, LS0 + R>(s, tw, m);
  }
}

// Bound of the lazy forward outputs with the fast butterflies: every forward pass
// (column then row, or one single pass) of the library ends below kFwdLazy * m.
constexpr u64 kFwdLazy = 70;

// Forward stages on the tile, by the modulus's class. Outputs are lazy (below
// kFwdLazy * m fast, 16m mid, 4m exact): reduce before use, or feed them to a
// reduction whose input bound allows it.
template <int LOGM, int LOGG, int P, int NT, bool ROW, int RM = 3>
__device__ __forceinline__ void tile_fwd(u64 *s, const ulonglong2 *tw, u64 m) {
  const int cls = mod_class(m);
  if (cls == CLS_FAST)
    tile_fwd_t<LOGM, LOGG, P, NT, ROW, RM, CLS_FAST>(s, tw, m);
  else if (cls == CLS_MID)
    tile_fwd_t<LOGM, LOGG, P, NT, ROW, RM, CLS_MID>(s, tw, m);
  else
    tile_fwd_t<LOGM, LOGG, P, NT, ROW, RM, CLS_EXACT>(s, tw, m);
}

// A lazy forward output of a modulus that is not fast, as a canonical residue.
__device__ __forceinline__ u64 fwd_canon(u64 y, u64 m, u64 mu, int cls) {
  return cls == CLS_EXACT ? csub(csub(y, 2 * m), m) : reduce_full(y, m, mu);
}

// Inverse stages LOGM-1..0 (bounds: see the butterflies).
template <int LOGM, int LOGG, int P, int NT, bool ROW, int RM, int CLS,
          int K = (LOGM + RM - 1) / RM - 1>
__device__ __forceinline__ void tile_inv_t(u64 *s, const ulonglong2 *tw, u64 m) {
  if constexpr (K >= 0 && LOGM > 0) {
    constexpr int LS0 = RM * K;
    constexpr int R = (LOGM - LS0) >= RM ? RM : (LOGM - LS0);
    ntt_round<LOGM, LOGG, P, NT, ROW, true, LS0, R, CLS>(s, tw, m);
    __syncthreads();
    tile_inv_t<LOGM, LOGG, P, NT, ROW, RM, CLS, K - 1>(s, tw, m);
  }
}

// Inverse stages by the modulus's class; inputs canonical. Outputs lazy (below 2^13 m
// fast, 8m mid, 2m exact): reduce with reduce_full or a Shoup scaling before use.
template <int LOGM, int LOGG, int P, int NT, bool ROW, int RM = 3>
__device__ __forceinline__ void tile_inv(u64 *s, const ulonglong2 *tw, u64 m) {
  const int cls = mod_class(m);
  if (cls == CLS_FAST)
    tile_inv_t<LOGM, LOGG, P, NT, ROW, RM, CLS_FAST>(s, tw, m);
  else if (cls == CLS_MID)
    tile_inv_t<LOGM, LOGG, P, NT, ROW, RM, CLS_MID>(s, tw, m);
  else
    tile_inv_t<LOGM, LOGG, P, NT, ROW, RM, CLS_EXACT>(s, tw, m);
}

}  // namespace ks
