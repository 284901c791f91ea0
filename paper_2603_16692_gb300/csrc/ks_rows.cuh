// The kernels of the two-pass sizes on the register-tile core (ks_core.cuh): the input and
// accumulator iNTTs, the basis conversions with the forward column pass, the key multiply,
// the ModDown row pass and the plain forward passes. One set of kernels per N serves every
// radix and column tile that a plan may name.
#pragma once
#include "ks_core.cuh"
#include "ks_kern.cuh"

namespace ks {
namespace kern {

// Row tile of N = 2^LOGN: GP threads, GR rows of N2 points.
template <int LOGN, int GP_ = 64>
struct RowGeo {
  static constexpr int LOGA = geo_loga(LOGN), LOGB = LOGN - LOGA;
  using SB = core::Sub<LOGB, core::row_rl(LOGN)>;
  static constexpr int N1 = 1 << LOGA, N2 = 1 << LOGB;
  static constexpr int GP = GP_, GR = GP / SB::T, TILE = GR * N2;
  static constexpr int WR = 32 / SB::T;      // rows of a warp
  static constexpr int RP = core::row_pitch<SB>();  // words of a row in shared memory
  static constexpr int TILEW = GR * RP;      // words of a tile
  static constexpr int TWR = N2 * GR;        // twiddle entries of a tile
  static constexpr int TW_BYTES = TWR * 16;
  static constexpr int GRID = N1 / GR;
  static_assert(GRID % 4 == 0, "tiles of a CTA");
  static_assert(SB::T <= 32, "a row inside a warp");
};

// CTAs of 128 threads per SM that the row kernels' registers leave room for: 64 registers
// at 8 points per thread, 80 at 16 (which spills at 64).
__host__ __device__ constexpr int row_blocks(int logn) { return core::row_rl(logn) == 3 ? 8 : 6; }

// The twiddle slab of (prime, row tile) by one bulk copy (see stage_tw); tw_ready waits.
template <class RG>
__device__ __forceinline__ void stage_row_tw(ulonglong2 *tws, const ulonglong2 *tab, int prime,
                                             int blk, u64 *bar) {
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_expect_tx(bar, RG::TW_BYTES);
    bulk_g2s(tws, tab + (((size_t)prime << RG::LOGB) << RG::LOGA) + (size_t)blk * RG::TWR,
             RG::TW_BYTES, bar);
  }
}

template <class RG>
__device__ __forceinline__ void row_fwd_cls(u64 *v, u64 *s, const ulonglong2 *tw, u64 m, int t,
                                            int cls) {
  if (cls == CLS_FAST)
    core::row_fwd<typename RG::SB, CLS_FAST>(v, s, tw, m, t);
  else if (cls == CLS_MID)
    core::row_fwd<typename RG::SB, CLS_MID>(v, s, tw, m, t);
  else
    core::row_fwd<typename RG::SB, CLS_EXACT>(v, s, tw, m, t);
}
template <class RG>
__device__ __forceinline__ void row_inv_cls(u64 *v, u64 *s, const ulonglong2 *tw, u64 m, int t,
                                            int cls) {
  if (cls == CLS_FAST)
    core::row_inv<typename RG::SB, CLS_FAST>(v, s, tw, m, t);
  else if (cls == CLS_MID)
    core::row_inv<typename RG::SB, CLS_MID>(v, s, tw, m, t);
  else
    core::row_inv<typename RG::SB, CLS_EXACT>(v, s, tw, m, t);
}

// Lane-linear 16-byte walk over a warp's own rows: pair k of lane l covers words
// 2 (l + 32 k) of the warp's WR rows (contiguous in global memory); calls f(k, word offset
// in the warp's rows, position in its shared rows).
template <class RG, class F>
__device__ __forceinline__ void warp_rows(F f) {
#pragma unroll
  for (int k = 0; k < RG::WR * RG::N2 / 64; ++k) {
    const int e = 2 * ((threadIdx.x & 31) + 32 * k);
    f(k, e, (e >> RG::LOGB) * RG::RP + core::row_pos(e & (RG::N2 - 1)));
  }
}

// A lane's pairs of the warp's rows at src, all in flight before the first is used. (A load
// in the loop that also stores is not moved above the store of the pair before, which may
// be its source: one round trip per pair. (2, 2^15, 10) 63.9 ->
// 62.3 us, (4, 2^16, 35) on tensor cores 316 -> 310. The accumulators' pairs loaded before
// the transform instead of after it: 311.)
template <class RG>
struct WarpPairs {
  ulonglong2 x[RG::WR * RG::N2 / 64];
  __device__ __forceinline__ void load(const u64 *src) {
    warp_rows<RG>([&](int k, int e, int) {
      x[k] = *reinterpret_cast<const ulonglong2 *>(src + e);
    });
  }
};

// The warp's rows of an inverse pass's input, into their shared rows; an input in host memory
// leaves its copy in device memory on the way. `paced` (large host inputs): one pair of a
// lane in flight at a time, since the reads share the CPU link with the previous
// operation's result, which is on the longer path: (1, 2^17, 4) 179.6 -> 175.1 us,
// (2, 2^17, 4) 171.8 -> 167.6, (2, 2^15, 10) 92.3 -> 91.7, against (4, 2^16, 20) 339 -> 345.
// Small inputs wait for latency instead and take all pairs at once ((1, 2^15, 1) 39.2 ->
// 35.8); the line is between 1.5 MB (62.7 -> 62.1) and 2.6 MB (89.5 -> 92.1).
constexpr int kPacedWords = 1 << 18;
template <class RG>
__device__ __forceinline__ void input_rows(u64 *ws, const u64 *src, u64 *copy, bool paced) {
  if (copy && paced) {
#pragma unroll 1
    for (int k = 0; k < RG::WR * RG::N2 / 64; ++k) {
      const int e = 2 * ((threadIdx.x & 31) + 32 * k);
      const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(src + e);
      *reinterpret_cast<ulonglong2 *>(copy + e) = x;
      *reinterpret_cast<ulonglong2 *>(ws + (e >> RG::LOGB) * RG::RP +
                                      core::row_pos(e & (RG::N2 - 1))) = x;
    }
    return;
  }
  WarpPairs<RG> in;
  in.load(src);
  warp_rows<RG>([&](int k, int, int p) { *reinterpret_cast<ulonglong2 *>(ws + p) = in.x[k]; });
  if (copy)
    warp_rows<RG>([&](int k, int e, int) { *reinterpret_cast<ulonglong2 *>(copy + e) = in.x[k]; });
}

// A value between the two inverse passes: the column pass starts from values below 4m
// (fast; the row pass leaves them below 2^10 m), or takes the row pass's bounds as they are
// (mid: 8m, exact: 2m). q = floor(x_hi floor(2^64 / m) / 2^32) is at most 3 below x / m when
// m > 2^32; smaller fast moduli take the full reduction. One 32x32 product for the quotient
// instead of a 64x64 one: six instructions a point against eighteen.
__device__ __forceinline__ u64 inv_between(u64 x, u64 m, u64 mu, int cls) {
  if (cls != CLS_FAST) return x;
  if (mu >> 32) return reduce_full(x, m, mu);
  return x - (u64)__umulhi((uint32_t)(x >> 32), (uint32_t)mu) * m;
}

// ---------------------------------------------------------------------------
// Inverse row pass: d -> v (which 0, one polynomial) or the P-limbs of acc -> vp (which 1,
// both polynomials, one group of 64 threads each, sharing the twiddle slab). Lazy output
// (inv_between), within the bounds that col_inv starts from. Bound by the integer pipe and the twiddle slab's traffic
// (16 bytes per point against 8 in and 8 out).
template <int LOGN>
__global__ void __launch_bounds__(128, row_blocks(LOGN))
    k_inv_row2(KArgs a, JobSet js, WsOff wo, int which) {
  using RG = RowGeo<LOGN>;
  using SB = typename RG::SB;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  const JobPtr &jp = js.j[blockIdx.z];
  const InttSet is = intt_set(a, jp, wo, which);
  const int o = threadIdx.x / RG::GP, tg = threadIdx.x % RG::GP;
  const int row = tg / SB::T, t = tg % SB::T, w0 = row / RG::WR * RG::WR;  // warp's first row
  const int ii = blockIdx.y, prime = is.prime_base + ii, blk = blockIdx.x, r0 = blk * RG::GR;
  u64 *tile = reinterpret_cast<u64 *>(raw + RG::TW_BYTES) + o * RG::TILEW;
  const ModInfo &mi = a.tab.mod[prime];
  const u64 m = mi.m, mu = mi.mu;
  constexpr size_t N = (size_t)1 << LOGN;
  stage_row_tw<RG>(tws, a.tab.twr_f, prime, RG::N1 / RG::GR - 1 - blk, &twbar);
  // (see inv_row_body: an input in host memory that the predecessor does not write is read
  // without waiting for it; it is waited for at the end)
  const bool host_in = which == 0 && jp.dsrc, ahead = host_in && jp.ahead;
  if (!ahead) pdl_wait(a.early);
  const size_t off = ((size_t)(r0 + w0) << RG::LOGB);
  const u64 *src = host_in ? jp.dsrc + (size_t)ii * N + off
                           : is.src + ((size_t)o * is.src_outer + ii) * N + off;
  u64 *ws = tile + w0 * RG::RP;
  input_rows<RG>(ws, src, host_in ? const_cast<u64 *>(jp.d) + (size_t)ii * N + off : nullptr,
                 (a.nq << LOGN) > kPacedWords);
  __syncthreads();  // the warp's rows, and the barrier's initialisation
  tw_ready<true>(&twbar, a.tab.err);
  u64 v[SB::E];
  u64 *s = tile + row * RG::RP;
  core::get_row<SB>(v, s, t);
  const int cls = mod_class(m);
  row_inv_cls<RG>(v, s, tws + (size_t)(RG::GR - 1 - row) * RG::N2, m, t, cls);
  u64 *d = is.dst + ((size_t)o * is.dst_outer + ii) * N + ((size_t)(r0 + row) << RG::LOGB);
#pragma unroll
  for (int u = 0; u < SB::E; ++u) d[(u << SB::LOGT) + t] = inv_between(v[u], m, mu, cls);
  if (ahead) pdl_wait(a.early);
  pdl_trigger();
}

// ---------------------------------------------------------------------------
// Inverse column pass, in place, with the per-limb scale; `pieces` writes the bf16 bytes
// of the result for the tensor-core conversion (ks_tc.cu) instead: the limb's columns in
// blocks of 2^tplog / N1, block after block; inside a block, point (y, g) at y * (columns per
// block) + g, 16 bytes (eight bf16) per point. Both polynomials of which = 1 run side by side.
template <int LOGN>
struct ColGeo {
  static constexpr int LOGA = geo_loga(LOGN), LOGB = LOGN - LOGA;
  static constexpr int N1 = 1 << LOGA, N2 = 1 << LOGB;
  static constexpr int RL = core::col_rl(LOGN), E = 1 << RL, LOGT = LOGA - RL;
  static constexpr int GC = 8;             // columns per tile: 64-byte row segments
  static constexpr int GP = GC << LOGT;    // threads of a tile
  static constexpr int TILEW = core::col_words<LOGA, GC, RL>();
  static constexpr int KL = core::col_rounds<LOGA, RL>() - 1;  // last round
  static constexpr int TW_BYTES = N1 * 16;
  static constexpr int GRID = N2 / GC;
};

template <int LOGN>
__global__ void __launch_bounds__(2 * ColGeo<LOGN>::GP, 768 / (2 * ColGeo<LOGN>::GP))
    k_inv_col2(KArgs a, JobSet js, WsOff wo, int which, int pieces) {
  using CG = ColGeo<LOGN>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  const JobPtr &jp = js.j[blockIdx.z];
  const InttSet is = intt_set(a, jp, wo, which);
  const int o = threadIdx.x / CG::GP, tg = threadIdx.x % CG::GP;
  const int g = tg % CG::GC, t = tg / CG::GC, c0 = blockIdx.x * CG::GC;
  const int ii = blockIdx.y, prime = is.prime_base + ii;
  u64 *tile = reinterpret_cast<u64 *>(raw + CG::TW_BYTES) + o * CG::TILEW;
  const u64 m = a.tab.mod[prime].m;
  if (threadIdx.x == 0) {
    mbar_init(&twbar, 1);
    mbar_expect_tx(&twbar, CG::TW_BYTES);
    bulk_g2s(tws, a.tab.twc_i + ((size_t)prime << CG::LOGA), CG::TW_BYTES, &twbar);
  }
  pdl_wait(a.early);
  u64 *d = is.dst + ((size_t)o * is.dst_outer + ii) * ((size_t)1 << LOGN);
  u64 v[CG::E];
#pragma unroll
  for (int r = 0; r < CG::E; ++r)
    v[r] = d[((size_t)core::ColRound<CG::LOGA, CG::RL, CG::KL>::point(t, r) << CG::LOGB) + c0 + g];
  const ulonglong2 sc = is.scale[ii];
  __syncthreads();  // the barrier's initialisation
  tw_ready<true>(&twbar, a.tab.err);
  const int cls = mod_class(m);
  auto sync = [] { __syncthreads(); };
  if (cls == CLS_FAST)
    core::col_inv<CG::LOGA, CG::RL, CG::GC, CLS_FAST, CG::KL>(v, tile, tws, m, t, g, sync);
  else if (cls == CLS_MID)
    core::col_inv<CG::LOGA, CG::RL, CG::GC, CLS_MID, CG::KL>(v, tile, tws, m, t, g, sync);
  else
    core::col_inv<CG::LOGA, CG::RL, CG::GC, CLS_EXACT, CG::KL>(v, tile, tws, m, t, g, sync);
#pragma unroll
  for (int u = 0; u < CG::E; ++u) v[u] = csub(shoup(v[u], sc.x, sc.y, m), m);
  const int col = c0 + g;
  if (pieces) {
    const size_t limb = which == 0 ? (size_t)ii : (size_t)o * a.np + ii;
    const int lgc = a.tc_tplog - CG::LOGA;
    u64 *pb = jp.ws + (which == 0 ? wo.pv : wo.ppv) + (limb << (LOGN + 1)) +
              2 * (((size_t)(col >> lgc) << a.tc_tplog) + (col & ((1 << lgc) - 1)));
#pragma unroll
    for (int u = 0; u < CG::E; ++u)
      *reinterpret_cast<uint4 *>(pb + ((size_t)((u << CG::LOGT) + t) << (lgc + 1))) =
          bf16_bytes(v[u]);
  } else {
#pragma unroll
    for (int u = 0; u < CG::E; ++u) d[((size_t)((u << CG::LOGT) + t) << CG::LOGB) + col] = v[u];
  }
  pdl_trigger();
}

// Terms whose middle products stay below 2^63 - 2^33 in the key multiply: 71 m + 2^33 each
// with lazy ext (below 70 m, m < 2^51), 2 m + 2^33 otherwise (m < 2^60); exact moduli fold
// every term.
__device__ __forceinline__ int mac_terms(int cls) {
  return cls == CLS_FAST ? 32 : cls == CLS_MID ? 3 : 1;
}

// Forward column tile: 8 columns, 8 points per thread.
template <int LOGN>
struct FwdColGeo {
  static constexpr int LOGA = geo_loga(LOGN), LOGB = LOGN - LOGA;
  static constexpr int N1 = 1 << LOGA, N2 = 1 << LOGB;
  static constexpr int RL = 3, E = 8, GC = 8, GP = GC * N1 / E;
  static constexpr int TILEW = core::col_words<LOGA, GC, RL>();
  static constexpr int TW_BYTES = N1 * 16;
  static constexpr int GRID = N2 / GC, SMEM = TW_BYTES + TILEW * 8;
};

// Fast basis conversion of a thread's eight points of a column (points C0::point(t, .) of the
// first forward round; src: the sources' limb 0 at the column) onto limb tgt: REDC(sum_i
// x_i c_i), canonical. PRO_UP: from digit dig's limbs of v; PRO_DOWN: from polynomial dig's
// P-limbs of vp. The sums are exact (Mac3), four points at a time.
template <int PRO, int LOGN>
__device__ __forceinline__ void bconv_points(u64 *v, const KArgs &a, int tgt, int dig,
                                             const u64 *src, int t, int cls) {
  constexpr int LOGA = geo_loga(LOGN), LOGB = LOGN - LOGA;
  using C0 = core::ColRound<LOGA, 3, 0>;
  const ModInfo &mi = a.tab.mod[tgt];
  const u64 m = mi.m;
  const int i0 = dig * (PRO == PRO_UP ? a.alpha : a.np);
  const int ns = PRO == PRO_UP ? min(a.nq, i0 + a.alpha) - i0 : a.np;
  const u64 *cst = PRO == PRO_UP ? a.tab.cup + ((size_t)dig * a.qp + tgt) * a.alpha
                                 : a.tab.cdown + (size_t)tgt * a.alpha;
  // run: terms of one reduction (their sum below m 2^64); fl: terms whose middle products
  // stay below 2^63 (source + m + 2^33 each), or 2^64 where the reduction folds them first
  const int run = PRO == PRO_UP ? a.run_up : a.run_down;
  const int fl = min(run, cls == CLS_FAST && run >= (1 << 13) ? 1 << 10 : run >= 16 ? 3 : 1);
  const int rcls = run < 16 ? CLS_EXACT : cls;  // a modulus or a source above 2^60
  const uint32_t inv = 0u - (uint32_t)mi.minv;
  src += (size_t)i0 << LOGN;
  constexpr int H = 4;  // points per batch (eight spill: (2, 2^15, 10) 63 -> 72 us)
#pragma unroll
  for (int h = 0; h < 8; h += H) {
    Mac3 s[H] = {};
    u64 x[H];
#pragma unroll
    for (int k = 0; k < H; ++k) x[k] = src[(size_t)C0::point(t, h + k) << LOGB];
    if (ns <= fl) {  // the usual case: one sum, no fold on the way
#pragma unroll 2
      for (int i = 0; i < ns; ++i) {
        const u64 c = __ldg(cst + i);
        u64 xn[H];
        if (i + 1 < ns) {  // the next limb's loads before this one's products
          const u64 *sn = src + ((size_t)(i + 1) << LOGN);
#pragma unroll
          for (int k = 0; k < H; ++k) xn[k] = sn[(size_t)C0::point(t, h + k) << LOGB];
        }
#pragma unroll
        for (int k = 0; k < H; ++k) s[k].add(x[k], c);
#pragma unroll
        for (int k = 0; k < H; ++k) x[k] = xn[k];
      }
#pragma unroll
      for (int k = 0; k < H; ++k) v[h + k] = mac_reduce(s[k], mi, m, inv, rcls);
    } else {
#pragma unroll
      for (int k = 0; k < H; ++k) v[h + k] = 0;
      int left = run, fold = fl;
#pragma unroll 1
      for (int i = 0; i < ns; ++i) {
        const u64 c = __ldg(cst + i);
        u64 xn[H];
        if (i + 1 < ns) {
          const u64 *sn = src + ((size_t)(i + 1) << LOGN);
#pragma unroll
          for (int k = 0; k < H; ++k) xn[k] = sn[(size_t)C0::point(t, h + k) << LOGB];
        }
#pragma unroll
        for (int k = 0; k < H; ++k) s[k].add(x[k], c);
        --left;
        if (left == 0 || i == ns - 1) {
          left = run;
          fold = fl;
#pragma unroll
          for (int k = 0; k < H; ++k) {
            v[h + k] = csub(v[h + k] + mac_reduce(s[k], mi, m, inv, rcls), m);
            s[k] = Mac3{};
          }
        } else if (--fold == 0) {
          fold = fl;
#pragma unroll
          for (int k = 0; k < H; ++k) s[k].fold();
        }
#pragma unroll
        for (int k = 0; k < H; ++k) x[k] = xn[k];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Forward column pass: the integer basis conversion of a task (PRO_UP, PRO_DOWN) or a plain
// load (PRO_LOAD, in place), then the first forward NTT pass on the thread's eight points.
// The conversion ends in registers; the tile in shared memory is only the NTT's exchange.
// Bound by the integer pipe.
template <int LOGN, int PRO>
__global__ void __launch_bounds__(FwdColGeo<LOGN>::GP, 768 / FwdColGeo<LOGN>::GP)
    k_fwd_col2(KArgs a, JobSet js, WsOff wo, Tasks tk, int buf) {
  using CG = FwdColGeo<LOGN>;
  using C0 = core::ColRound<CG::LOGA, CG::RL, 0>;
  using CL = core::ColRound<CG::LOGA, CG::RL, core::col_rounds<CG::LOGA, CG::RL>() - 1>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *tile = reinterpret_cast<u64 *>(raw + CG::TW_BYTES);
  const u64 *src;
  u64 *dst;
  fwd_bufs<PRO>(js.j[blockIdx.z], wo, buf, src, dst);
  const uint32_t w = decode(a, tk, blockIdx.y);
  const int tgt = task_limb(w), dig = task_dig(w);
  const int g = threadIdx.x % CG::GC, t = threadIdx.x / CG::GC, c0 = blockIdx.x * CG::GC;
  if (threadIdx.x == 0) {
    mbar_init(&twbar, 1);
    mbar_expect_tx(&twbar, CG::TW_BYTES);
    bulk_g2s(tws, a.tab.twc_f + ((size_t)tgt << CG::LOGA), CG::TW_BYTES, &twbar);
  }
  const ModInfo &mi = a.tab.mod[tgt];
  const u64 m = mi.m;
  const int cls = mod_class(m);
  dst += ((size_t)task_slot(w) << LOGN) + c0 + g;
  u64 v[CG::E];
  if constexpr (PRO == PRO_LOAD) {
    pdl_wait(a.early);
#pragma unroll
    for (int r = 0; r < CG::E; ++r) v[r] = dst[(size_t)C0::point(t, r) << CG::LOGB];
  } else {
    pdl_wait(a.early);
    bconv_points<PRO, LOGN>(v, a, tgt, dig, src + c0 + g, t, cls);
  }
  __syncthreads();  // the barrier's initialisation
  tw_ready<true>(&twbar, a.tab.err);
  auto sync = [] { __syncthreads(); };
  if (cls == CLS_FAST)
    core::col_fwd<CG::LOGA, CG::RL, CG::GC, CLS_FAST, 0>(v, tile, tws, m, t, g, sync);
  else if (cls == CLS_MID)
    core::col_fwd<CG::LOGA, CG::RL, CG::GC, CLS_MID, 0>(v, tile, tws, m, t, g, sync);
  else
    core::col_fwd<CG::LOGA, CG::RL, CG::GC, CLS_EXACT, 0>(v, tile, tws, m, t, g, sync);
#pragma unroll
  for (int r = 0; r < CG::E; ++r) dst[(size_t)CL::point(t, r) << CG::LOGB] = v[r];
  pdl_trigger();
}

// ---------------------------------------------------------------------------
// Plain forward row pass (keygen, unfused plans): canonical result back in place.
template <int LOGN>
__global__ void __launch_bounds__(64)
    k_row_store2(KArgs a, JobSet js, WsOff wo, Tasks tk, int buf) {
  using RG = RowGeo<LOGN>;
  using SB = typename RG::SB;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *tile = reinterpret_cast<u64 *>(raw + RG::TW_BYTES);
  const int row = threadIdx.x / SB::T, t = threadIdx.x % SB::T, w0 = row / RG::WR * RG::WR;
  const u64 *src;
  u64 *dst;
  fwd_bufs<PRO_LOAD>(js.j[blockIdx.z], wo, buf, src, dst);
  const uint32_t w = decode(a, tk, blockIdx.y);
  const int p = task_limb(w), blk = blockIdx.x, r0 = blk * RG::GR;
  const ModInfo &mi = a.tab.mod[p];
  const u64 m = mi.m, mu = mi.mu;
  stage_row_tw<RG>(tws, a.tab.twr_f, p, blk, &twbar);
  pdl_wait(a.early);
  u64 *b = dst + ((size_t)task_slot(w) << LOGN);
  u64 v[SB::E];
#pragma unroll
  for (int u = 0; u < SB::E; ++u)
    v[u] = b[((size_t)(r0 + row) << RG::LOGB) + (u << SB::LOGT) + t];
  __syncthreads();
  tw_ready<true>(&twbar, a.tab.err);
  u64 *s = tile + row * RG::RP;
  row_fwd_cls<RG>(v, s, tws + row * RG::N2, m, t, mod_class(m));
  __syncwarp();
  core::put_row<SB>(s, v, t);
  __syncwarp();
  const u64 *ws = tile + w0 * RG::RP;
  u64 *o = b + ((size_t)(r0 + w0) << RG::LOGB);
  warp_rows<RG>([&](int, int e, int q) {
    ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(ws + q);
    x.x = reduce_full(x.x, m, mu);
    x.y = reduce_full(x.y, m, mu);
    *reinterpret_cast<ulonglong2 *>(o + e) = x;
  });
  pdl_trigger();
}

// ---------------------------------------------------------------------------
// Key multiply (TASK_TARGET): one CTA = one row tile of one target limb t, all its digits:
//   acc_c[t] (+)= sum_j ext_j[t] * evk[j][c][t],  c = 0, 1.
// Groups of kKmGp threads transform one digit's tile each, side by side on one twiddle slab,
// and leave ext in shared memory; after one barrier every thread multiplies its points by
// the key words of all digits (read once, 16 bytes a lane, pulled into L2 by the TMA unit
// while the digits are transformed) with exact 128-bit sums and one REDC per output word.
// The CTA's own digit (t's limb inside the digit) is the input itself, put in Montgomery
// form. Up to `ds` digits fit at a time; more are taken in turns, the accumulators
// re-read.
constexpr int kKmDigits = 10;   // most digits of a tile held in shared memory
constexpr int kKmGroups = 4;    // most groups of threads (one tile each)

// The multiply phase of a key multiply: for every point e of a tile (`words` points),
//   acc_c[e] (+)= sum_j ext_j[e] * key_jc[e],  c = 0, 1, over n digits.
// ext: digit tiles in shared memory, `tilew` words apart, rows of 2^LOGB points at a pitch
// of RP; kp: the tile's key words of digit 0, polynomial 0, polynomials cst words apart
// (digits 2 cst); o: accumulators, polynomials oc1 words apart; first: write, else add (FIRST: always write,
// without the old accumulators' registers).
// One loop of (pair of points, digit) steps. The next step's key words (and at a new pair
// the old accumulators) are loaded before a step's products, the first ones before
// ready(), the barrier after which ext may be read.
template <int LOGB, int RP, bool FIRST, class READY>
__device__ __forceinline__ void mac_tile(const ModInfo &mi, const u64 *ext, int tilew, int n,
                                         int words, const u64 *kp, size_t cst, u64 *o, size_t oc1,
                                         bool first, int cls, READY ready) {
  first = first || FIRST;
  const u64 m = mi.m, pol = l2_stream();
  const uint32_t inv = 0u - (uint32_t)mi.minv;
  const int bd = blockDim.x, fl = mac_terms(cls);
  kp += 2 * threadIdx.x;
  o += 2 * threadIdx.x;
  ulonglong2 na = {}, nb = {}, no0 = {}, no1 = {}, old0 = {}, old1 = {};
  if (2 * threadIdx.x < words) {
    na = ldg_pol(reinterpret_cast<const ulonglong2 *>(kp), pol);
    nb = ldg_pol(reinterpret_cast<const ulonglong2 *>(kp + cst), pol);
    if (!first) {
      no0 = *reinterpret_cast<const ulonglong2 *>(o);
      no1 = *reinterpret_cast<const ulonglong2 *>(o + oc1);
    }
  }
  ready();
  Mac3 s[4] = {};
  int jj = 0, fold = fl;
  auto pos = [&](int e) { return ext + (e >> LOGB) * RP + core::row_pos(e & ((1 << LOGB) - 1)); };
  const u64 *yp = pos(2 * threadIdx.x);
  for (int e = 2 * threadIdx.x; e < words;) {
    const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(yp);
    yp += tilew;
    const ulonglong2 ka = na, kb = nb;
    if (jj == 0) old0 = no0, old1 = no1;
    const bool last = jj == n - 1;
    kp += 2 * cst;
    if (last) kp += 2 * bd - 2 * cst * n;
    if (!last || e + 2 * bd < words) {
      na = ldg_pol(reinterpret_cast<const ulonglong2 *>(kp), pol);
      nb = ldg_pol(reinterpret_cast<const ulonglong2 *>(kp + cst), pol);
      if (last && !first) {
        no0 = *reinterpret_cast<const ulonglong2 *>(o + 2 * bd);
        no1 = *reinterpret_cast<const ulonglong2 *>(o + 2 * bd + oc1);
      }
    }
    s[0].add(y.x, ka.x);
    s[1].add(y.y, ka.y);
    s[2].add(y.x, kb.x);
    s[3].add(y.y, kb.y);
    if (last) {
      u64 r[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        r[i] = mac_reduce(s[i], mi, m, inv, cls);
        s[i] = Mac3{};
      }
      if (!first) {
        r[0] = addmod(r[0], old0.x, m);
        r[1] = addmod(r[1], old0.y, m);
        r[2] = addmod(r[2], old1.x, m);
        r[3] = addmod(r[3], old1.y, m);
      }
      *reinterpret_cast<ulonglong2 *>(o) = make_ulonglong2(r[0], r[1]);
      *reinterpret_cast<ulonglong2 *>(o + oc1) = make_ulonglong2(r[2], r[3]);
      o += 2 * bd;
      e += 2 * bd;
      yp = pos(e);
      jj = 0;
      fold = fl;
    } else {
      ++jj;
      if (--fold == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i].fold();
        fold = fl;
      }
    }
  }
}

// Own digit's tile: the warp's rows of the input in Montgomery form, into their shared rows.
template <class RG>
__device__ __forceinline__ void own_rows(u64 *ws, const u64 *dt, const ModInfo &mi, bool lazy) {
  const u64 m = mi.m, r1 = mi.r1, r1s = mi.r1s;
  WarpPairs<RG> in;
  in.load(dt);
  warp_rows<RG>([&](int k, int, int p) {
    ulonglong2 x = in.x[k];
    if (lazy) {
      x.x = shoup4(x.x, r1, r1s, m);  // [0, 4m)
      x.y = shoup4(x.y, r1, r1s, m);
    } else {
      x.x = csub(shoup(x.x, r1, r1s, m), m);
      x.y = csub(shoup(x.y, r1, r1s, m), m);
    }
    *reinterpret_cast<ulonglong2 *>(ws + p) = x;
  });
}

// A tile is one warp's rows (one row of 256 or 512 points, two of 128): small CTAs, so that
// several of them mix their transform and multiply phases on an SM (tiles of two warps:
// (4, 2^16, 35) 346 -> 341 us, (8, 2^16, 15) 239 -> 234).
constexpr int kKmGp = 32;

template <int LOGN, bool FIRST>
__global__ void __launch_bounds__(kKmGp * kKmGroups, 768 / (kKmGp * kKmGroups))
    k_keymult2(KArgs a, JobSet js, WsOff wo, Tasks tk, int ds) {
  using RG = RowGeo<LOGN, kKmGp>;
  using SB = typename RG::SB;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *ext = reinterpret_cast<u64 *>(raw + RG::TW_BYTES);
  const JobPtr &jp = js.j[blockIdx.z];
  const int grp = threadIdx.x / RG::GP, ngrp = blockDim.x / RG::GP, tg = threadIdx.x % RG::GP;
  const int row = tg / SB::T, t = tg % SB::T, w0 = row / RG::WR * RG::WR;
  // targets in reverse: the P-limb targets, listed last, transform every digit (a Q-limb
  // target's own digit needs no transform), so they start first
  const int tgt = tk.t0 + (gridDim.y - 1 - blockIdx.y);
  const ModInfo &mi = a.tab.mod[tgt];
  const u64 m = mi.m;
  const int blk = blockIdx.x, off0 = blk * RG::TILE;
  const int od = tgt < a.nq ? tgt / a.alpha : -1;  // the target's own digit
  const int nd = tk.j1 - tk.j0;
  // the tile's key words: digit j, polynomial c at (2j + c) eqp N words further
  const u64 *evk = jp.evk + ((size_t)(tgt < a.nq ? tgt : a.epb + (tgt - a.nq)) << LOGN) + off0;
  for (int k = threadIdx.x; k < 2 * nd; k += blockDim.x)
    prefetch_l2(evk + ((size_t)((2 * tk.j0 + k) * a.eqp) << LOGN), RG::TILE * 8);
  stage_row_tw<RG>(tws, a.tab.twr_f, tgt, blk, &twbar);
  const int cls = mod_class(m);
  // ext stays lazy when the exact digit sum of its products fits one reduction
  const bool lazy = cls == CLS_FAST && __umul64hi(kFwdLazy * min(nd, ds), m) == 0;
  pdl_wait(a.early);
  __syncthreads();  // the twiddle barrier's initialisation
  for (int c0 = tk.j0; c0 < tk.j1; c0 += ds) {
    const int n = min(ds, tk.j1 - c0);
    const int oc = od - c0;  // the own digit's index in this turn, if any
    const bool has = oc >= 0 && oc < n;
    for (int jj = grp; jj < n; jj += ngrp) {
      // the digits to transform first, the own digit (cheap) last
      const int jx = !has ? jj : jj == n - 1 ? oc : jj < oc ? jj : jj + 1;
      u64 *ex = ext + jx * RG::TILEW;
      if (has && jx == oc) {
        const u64 *dt = jp.d + ((size_t)tgt << LOGN) + off0 + (w0 << RG::LOGB);
        own_rows<RG>(ex + w0 * RG::RP, dt, mi, lazy);
        continue;
      }
      const int j = c0 + jx;
      const u64 *src = jp.ws + wo.tmp +
                       ((size_t)(j * tk.sm.sj + tgt * tk.sm.st + tk.sm.base) << LOGN) + off0 +
                       (row << RG::LOGB) + t;
      u64 v[SB::E];
#pragma unroll
      for (int u = 0; u < SB::E; ++u) v[u] = src[u << SB::LOGT];
      tw_ready<true>(&twbar, a.tab.err);
      u64 *s = ex + row * RG::RP;
      row_fwd_cls<RG>(v, s, tws + row * RG::N2, m, t, cls);
      if (!lazy) {
        const u64 mu = mi.mu;
#pragma unroll
        for (int r = 0; r < SB::E; ++r) v[r] = fwd_canon(v[r], m, mu, cls);
      }
      __syncwarp();
      core::put_row<SB>(s, v, t);
    }
    mac_tile<RG::LOGB, RG::RP, FIRST>(
        mi, ext, RG::TILEW, n, RG::TILE, evk + (((size_t)(2 * c0) * a.eqp) << LOGN),
        (size_t)a.eqp << LOGN, jp.ws + wo.acc + ((size_t)tgt << LOGN) + off0,
        (size_t)a.qp << LOGN, tk.first && c0 == tk.j0, cls,
        [&] {
          __syncthreads();
          tw_ready<true>(&twbar, a.tab.err);  // (a CTA with no digit to transform, too)
        });
    if (c0 + ds < tk.j1) __syncthreads();  // ext is free for the next turn
  }
  pdl_trigger();
}

// The final scaling of a warp's rows: out = (acc - z) P^-1 (+ addend) at word offset ob of the
// output, z the NTT's lazy values in ws: below kFwdLazy * m (fast butterflies) or, after one
// conditional subtraction, below 8m (mid) or 2m (exact); acc + zb - z is then positive and
// below (kFwdLazy + 1) m, 9m or 3m < 2^64, and the Shoup product by P^-1 takes any word.
// paced (results to host memory, see input_rows): a pair at a time, so that the stores to the
// CPU link spread over the kernel: (2, 2^15, 10) 91.7 -> 90.3 us, (2, 2^16, 4) 88.7 -> 87.0,
// (2, 2^17, 4) the same, against (4, 2^16, 20) 345 -> 348.
template <class RG>
__device__ __forceinline__ void scale_rows(const JobPtr &jp, int c, const u64 *ws,
                                           const u64 *ac, size_t ob, const ulonglong2 &pv, u64 m,
                                           int cls, bool paced) {
  const bool fast = cls == CLS_FAST;
  const u64 zs = cls == CLS_MID ? 8 * m : 2 * m, zb = fast ? kFwdLazy * m : zs;
  auto word = [&](u64 z, u64 x) {
    return csub(shoup(x + zb - (fast ? z : csub(z, zs)), pv.x, pv.y, m), m);
  };
  if (paced) {  // (without addend)
#pragma unroll 1
    for (int k = 0; k < RG::WR * RG::N2 / 64; ++k) {
      const int e = 2 * ((threadIdx.x & 31) + 32 * k);
      const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(
          ws + (e >> RG::LOGB) * RG::RP + core::row_pos(e & (RG::N2 - 1)));
      const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(ac + e);
      *reinterpret_cast<ulonglong2 *>(jp.out + ob + e) =
          make_ulonglong2(word(z.x, x.x), word(z.y, x.y));
    }
    return;
  }
  WarpPairs<RG> acc;
  acc.load(ac);
  if ((jp.addmask >> c) & 1) {
    WarpPairs<RG> y;
    y.load(jp.add + ob);
    warp_rows<RG>([&](int k, int e, int q) {
      const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(ws + q);
      ulonglong2 r;
      r.x = addmod(word(z.x, acc.x[k].x), y.x[k].x, m);
      r.y = addmod(word(z.y, acc.x[k].y), y.x[k].y, m);
      *reinterpret_cast<ulonglong2 *>(jp.out + ob + e) = r;
    });
  } else {
    warp_rows<RG>([&](int k, int e, int q) {
      const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(ws + q);
      *reinterpret_cast<ulonglong2 *>(jp.out + ob + e) =
          make_ulonglong2(word(z.x, acc.x[k].x), word(z.y, acc.x[k].y));
    });
  }
}

// ---------------------------------------------------------------------------
// ModDown row pass with the final scaling (TASK_DOWN1):
//   out_c[i] = (acc_c[i] - NTT(BConv_{P->Q}(c))[i]) * P^-1 mod q_i (+ addend),
// the two polynomials of limb i side by side in two groups of 64 threads that share the
// twiddle slab; each warp finishes its own rows (no block barrier after the start).
template <int LOGN>
__global__ void __launch_bounds__(128, row_blocks(LOGN))
    k_moddown2(KArgs a, JobSet js, WsOff wo, Tasks tk) {
  using RG = RowGeo<LOGN>;
  using SB = typename RG::SB;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  const JobPtr &jp = js.j[blockIdx.z];
  // host-buffer operation: see k_fwd_row_moddown
  if (jp.dsrc) pdl_trigger();
  const int c = threadIdx.x / RG::GP, tg = threadIdx.x % RG::GP;
  const int row = tg / SB::T, t = tg % SB::T, w0 = row / RG::WR * RG::WR;
  const uint32_t w = decode(a, tk, blockIdx.y);
  const int i = task_limb(w), blk = blockIdx.x, r0 = blk * RG::GR;
  u64 *tile = reinterpret_cast<u64 *>(raw + RG::TW_BYTES) + c * RG::TILEW;
  const u64 m = a.tab.mod[i].m;
  const ulonglong2 pv = a.tab.pinv[i];
  constexpr size_t N = (size_t)1 << LOGN;
  stage_row_tw<RG>(tws, a.tab.twr_f, i, blk, &twbar);
  const int cls = mod_class(m);
  pdl_wait(a.early);
  const size_t woff = (size_t)(r0 + w0) << RG::LOGB;  // the warp's rows
  const u64 *ac = jp.ws + wo.acc + ((size_t)c * a.qp + i) * N + woff;
  u64 v[SB::E];
  {
    const u64 *src = jp.ws + wo.tmp2 + (size_t)(task_slot(w) + c * tk.span) * N +
                     ((size_t)(r0 + row) << RG::LOGB) + t;
#pragma unroll
    for (int u = 0; u < SB::E; ++u) v[u] = src[u << SB::LOGT];
  }
  if ((threadIdx.x & 31) == 0) prefetch_l2(ac, RG::WR * RG::N2 * 8);
  __syncthreads();  // the twiddle barrier's initialisation
  tw_ready<true>(&twbar, a.tab.err);
  u64 *s = tile + row * RG::RP;
  row_fwd_cls<RG>(v, s, tws + row * RG::N2, m, t, cls);
  __syncwarp();
  core::put_row<SB>(s, v, t);
  __syncwarp();
  const u64 *ws = tile + w0 * RG::RP;
  scale_rows<RG>(jp, c, ws, ac, ((size_t)c * a.nq + i) * N + woff, pv, m, cls,
                 jp.dsrc && !jp.addmask && (a.nq << LOGN) > kPacedWords);
  pdl_trigger();
}

// ---------------------------------------------------------------------------
// Launchers of one two-pass N.
template <int LOGN>
struct RowFns {
  using RG = RowGeo<LOGN>;
  using KG = RowGeo<LOGN, kKmGp>;  // the key multiply's tile
  using CG = ColGeo<LOGN>;
  using FG = FwdColGeo<LOGN>;
  static constexpr int smem_row(int tiles) { return RG::TW_BYTES + tiles * RG::TILEW * 8; }
  static constexpr int smem_km(int ds) { return KG::TW_BYTES + ds * KG::TILEW * 8; }
  static constexpr int smem_col(int tiles) { return CG::TW_BYTES + tiles * CG::TILEW * 8; }

  static cudaError_t prepare() {
    cudaError_t e;
    if ((e = smem_attr(k_inv_row2<LOGN>, smem_row(2)))) return e;
    if ((e = smem_attr(k_inv_col2<LOGN>, smem_col(2)))) return e;
    if ((e = smem_attr(k_fwd_col2<LOGN, PRO_LOAD>, FG::SMEM))) return e;
    if ((e = smem_attr(k_fwd_col2<LOGN, PRO_UP>, FG::SMEM))) return e;
    if ((e = smem_attr(k_fwd_col2<LOGN, PRO_DOWN>, FG::SMEM))) return e;
    if ((e = smem_attr(k_row_store2<LOGN>, smem_row(1)))) return e;
    if ((e = smem_attr(k_keymult2<LOGN, true>, smem_km(kKmDigits)))) return e;
    if ((e = smem_attr(k_keymult2<LOGN, false>, smem_km(kKmDigits)))) return e;
    return smem_attr(k_moddown2<LOGN>, smem_row(2));
  }
  static cudaError_t intt_row(const ks_context *c, const JobSet &js, const WsOff &wo, int which,
                              cudaStream_t s) {
    const int inner = which == 0 ? c->nq : c->np, tiles = which + 1;
    if (inner == 0 || js.n == 0) return cudaSuccess;
    return launch_rule(k_inv_row2<LOGN>, dim3(RG::GRID, inner, js.n), dim3(RG::GP * tiles),
                      smem_row(tiles), s, c, js, wo, which);
  }
  static cudaError_t col(const ks_context *c, const JobSet &js, const WsOff &wo, int which,
                         int pieces, cudaStream_t s) {
    const int inner = which == 0 ? c->nq : c->np, tiles = which + 1;
    if (inner == 0 || js.n == 0) return cudaSuccess;
    KArgs a = args_of(c);
    const dim3 grid(CG::GRID, inner, js.n), block(CG::GP * tiles);
    // writing bytes, the tensor-core kernel follows: one CTA per SM, which cannot crowd the
    // SMs that this launch leaves empty ((4, 2^16, 35) 324 -> 317 us)
    a.early = pieces || early_rule((size_t)grid.x * grid.y * grid.z * block.x);
    return launch_pdl(k_inv_col2<LOGN>, grid, block, smem_col(tiles), s, a, js, wo, which, pieces);
  }
  static cudaError_t intt_col(const ks_context *c, const JobSet &js, const WsOff &wo, int which,
                              cudaStream_t s) {
    return col(c, js, wo, which, 0, s);
  }
  static cudaError_t intt_col_tc(const ks_context *c, const JobSet &js, const WsOff &wo,
                                 int which, cudaStream_t s) {
    return col(c, js, wo, which, 1, s);
  }
  template <int PRO>
  static cudaError_t fwd_col(const ks_context *c, const JobSet &js, const WsOff &wo,
                             const Tasks &tk, int buf, cudaStream_t s) {
    const int n = count_tasks(c, tk);
    if (n == 0 || js.n == 0) return cudaSuccess;
    return launch_rule(k_fwd_col2<LOGN, PRO>, dim3(FG::GRID, n, js.n), dim3(FG::GP), FG::SMEM, s,
                      c, js, wo, tk, buf);
  }
  static cudaError_t modup_col(const ks_context *c, const JobSet &js, const WsOff &wo,
                               const Tasks &tk, cudaStream_t s) {
    return fwd_col<PRO_UP>(c, js, wo, tk, BUF_TMP, s);
  }
  static cudaError_t moddown_col(const ks_context *c, const JobSet &js, const WsOff &wo,
                                 const Tasks &tk, cudaStream_t s) {
    return fwd_col<PRO_DOWN>(c, js, wo, tk, BUF_TMP2, s);
  }
  static cudaError_t ntt_col(const ks_context *c, const JobSet &js, const WsOff &wo,
                             const Tasks &tk, int buf, cudaStream_t s) {
    return fwd_col<PRO_LOAD>(c, js, wo, tk, buf, s);
  }
  static cudaError_t modup_row(const ks_context *c, const JobSet &js, const WsOff &wo,
                               const Tasks &tk, cudaStream_t s) {
    const int n = count_tasks(c, tk), nd = tk.j1 - tk.j0;
    if (n == 0 || js.n == 0 || nd < 1) return cudaSuccess;
    const int turns = (nd + kKmDigits - 1) / kKmDigits, ds = (nd + turns - 1) / turns;
    const dim3 grid(KG::GRID, n, js.n), block(KG::GP * std::min(ds, kKmGroups));
    if (tk.first && turns == 1)
      return launch_rule(k_keymult2<LOGN, true>, grid, block, smem_km(ds), s, c, js, wo, tk, ds);
    return launch_rule(k_keymult2<LOGN, false>, grid, block, smem_km(ds), s, c, js, wo, tk, ds);
  }
  static cudaError_t moddown_row(const ks_context *c, const JobSet &js, const WsOff &wo,
                                 const Tasks &tk, cudaStream_t s) {
    const int n = count_tasks(c, tk);
    if (n == 0 || js.n == 0) return cudaSuccess;
    return launch_rule(k_moddown2<LOGN>, dim3(RG::GRID, n, js.n), dim3(RG::GP * 2), smem_row(2), s,
                      c, js, wo, tk);
  }
  static cudaError_t ntt_row(const ks_context *c, const JobSet &js, const WsOff &wo,
                             const Tasks &tk, int buf, cudaStream_t s) {
    const int n = count_tasks(c, tk);
    if (n == 0 || js.n == 0) return cudaSuccess;
    return launch_rule(k_row_store2<LOGN>, dim3(RG::GRID, n, js.n), dim3(RG::GP), smem_row(1), s,
                      c, js, wo, tk, buf);
  }
  static const LaunchTable &table() {
    static const LaunchTable t = {&prepare,     &count_tasks, &intt_row,  &intt_col,
                                  &intt_col_tc, &modup_col,   &modup_row, &moddown_col,
                                  &moddown_row, &ntt_col,     &ntt_row};
    return t;
  }
};

// Launchers of a single-pass size (N <= 2^11): the shared-memory tile rounds of radix RL.
template <int LOGN, int RL>
struct LaunchOne {
  using GTR = GeoT<LOGN, RL, 1>;

  static cudaError_t prepare() {
    cudaError_t e;
    if ((e = smem_attr(k_inv_row<LOGN, RL>, GTR::SMEM_ROW))) return e;
    if ((e = smem_attr(k_fwd_row_store<LOGN, RL>, GTR::SMEM_ROW))) return e;
    if ((e = smem_attr(k_fwd_row_keymult<LOGN, RL, PRO_UP>, GTR::SMEM_ROW))) return e;
    return smem_attr(k_fwd_row_moddown<LOGN, RL, PRO_DOWN>, GTR::SMEM_ROW);
  }
  static cudaError_t intt_row(const ks_context *c, const JobSet &js, const WsOff &wo, int which,
                              cudaStream_t s) {
    const int inner = which == 0 ? c->nq : c->np;
    if (inner == 0 || js.n == 0) return cudaSuccess;
    // the accumulator P-limbs hold two polynomials: one CTA each (a launch is a few CTAs)
    return launch_pdl(k_inv_row<LOGN, RL>, dim3(1, inner << which, js.n), dim3(GTR::NT),
                      GTR::SMEM_ROW, s, args_of(c), js, wo, which, which);
  }
  static cudaError_t no_col(const ks_context *, const JobSet &, const WsOff &, int,
                            cudaStream_t) {
    return cudaSuccess;
  }
  static cudaError_t no_col_task(const ks_context *, const JobSet &, const WsOff &,
                                 const Tasks &, cudaStream_t) {
    return cudaSuccess;
  }
  static cudaError_t no_ntt_col(const ks_context *, const JobSet &, const WsOff &,
                                const Tasks &, int, cudaStream_t) {
    return cudaSuccess;
  }
  static cudaError_t modup_row(const ks_context *c, const JobSet &js, const WsOff &wo,
                               const Tasks &tk, cudaStream_t s) {
    const int n = count_tasks(c, tk);
    if (n == 0 || js.n == 0) return cudaSuccess;
    return launch_pdl(k_fwd_row_keymult<LOGN, RL, PRO_UP>, dim3(1, n, js.n), dim3(GTR::NT),
                      GTR::SMEM_ROW, s, args_of(c), js, wo, tk);
  }
  static cudaError_t moddown_row(const ks_context *c, const JobSet &js, const WsOff &wo,
                                 const Tasks &tk, cudaStream_t s) {
    const int n = count_tasks(c, tk);
    if (n == 0 || js.n == 0) return cudaSuccess;
    return launch_pdl(k_fwd_row_moddown<LOGN, RL, PRO_DOWN>, dim3(1, n, js.n), dim3(GTR::NT),
                      GTR::SMEM_ROW, s, args_of(c), js, wo, tk);
  }
  static cudaError_t ntt_row(const ks_context *c, const JobSet &js, const WsOff &wo,
                             const Tasks &tk, int buf, cudaStream_t s) {
    const int n = count_tasks(c, tk);
    if (n == 0 || js.n == 0) return cudaSuccess;
    return launch_pdl(k_fwd_row_store<LOGN, RL>, dim3(1, n, js.n), dim3(GTR::NT), GTR::SMEM_ROW,
                      s, args_of(c), js, wo, tk, buf);
  }
  static const LaunchTable &table() {
    static const LaunchTable t = {&prepare,     &count_tasks, &intt_row,    &no_col,
                                  &no_col,      &no_col_task, &modup_row,   &no_col_task,
                                  &moddown_row, &no_ntt_col,  &ntt_row};
    return t;
  }
};

}  // namespace kern
}  // namespace ks
