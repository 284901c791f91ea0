// The steps of a KeySwitch as one kernel each for small N (2^12, 2^13; the inverse
// transform alone at 2^14): a cluster of
// eight CTAs holds a whole limb, a CTA an eighth of its columns in the column pass and an
// eighth of its rows in the row pass, and the points change hands through distributed
// shared memory between the two. Against the two kernels per step of the general path this
// takes out four launches with their fill and drain (more than the arithmetic of a pass at
// these sizes) and the ModUp and ModDown intermediates' trip through L2. Bound by latency:
// one or two warps per scheduler. (2, 2^12, 3): 27.9 us against 32.1 on the general kernels
// and 67.5 on one CTA per limb; where the line lies: fused_rule in ks_api.cu. The inverse
// transform is the faster form at every limb count up to 2^14, in front of the general
// kernels too ((7, 2^14, 30) 119.9 -> 113.6 us, (6, 2^13, 44) 85.3 -> 83.6), and the slower
// one at 2^15 ((10, 2^15, 33) 256 -> 276 us; clusters of 16: 271).
//   k_fu_inv    rows, columns and scale of one limb's iNTT (input limbs, or one polynomial's
//               P-limb of the accumulators)
//   k_fu_up     one target limb: per digit basis conversion, columns, rows; then the key
//               multiply over all digits
//   k_fu_down   one output limb of one polynomial: basis conversion, columns, rows, scaling
// One cluster barrier separates the passes (and one at the start, so that every CTA of the
// cluster runs before its shared memory is written).
#pragma once
#include "ks_rows.cuh"

namespace ks {
namespace kern {

constexpr int kFuC = 8;  // CTAs of a cluster (the portable maximum)
constexpr int kFuThreads = 512;

template <int LOGN>
struct FuGeo {
  static constexpr int LOGA = geo_loga(LOGN), LOGB = LOGN - LOGA;
  using SB = core::Sub<LOGB, 3>;
  static constexpr int N1 = 1 << LOGA, N2 = 1 << LOGB;
  static constexpr int RC = N1 / kFuC, CC = N2 / kFuC;  // rows and columns of a CTA
  static constexpr int PTS = RC * N2, NT = PTS / 8;     // points, threads (8 points each)
  static constexpr int T1 = N1 / 8, T2 = N2 / 8;        // threads of a column, of a row
  static constexpr int WR = 32 / T2;                    // rows of a warp
  static constexpr int RP = core::row_pitch<SB>(), ROWW = RC * RP;
  static constexpr int COLW = core::col_words<LOGA, CC, 3>();
  static constexpr int KL = core::col_rounds<LOGA, 3>() - 1;
  using C0 = core::ColRound<LOGA, 3, 0>;
  using CL = core::ColRound<LOGA, 3, KL>;
  static constexpr int TW_BYTES = N1 * 16 + PTS * 16;  // column table, the CTA's row slabs
  static_assert(SB::T == T2 && T2 <= 32 && RC * T2 == NT && CC * T1 == NT && RC % 8 == 0 &&
                    NT % 32 == 0 && NT <= kFuThreads,
                "a cluster of eight CTAs per limb");
  static constexpr int smem_inv() { return TW_BYTES + (ROWW + COLW) * 8; }
  static constexpr int smem_up(int digits, int groups) {
    return TW_BYTES + (digits * ROWW + groups * COLW) * 8;
  }
};

__device__ __forceinline__ uint32_t cluster_map(const void *p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_st(uint32_t addr, u64 x) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(x) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// The column table of `prime` and the row slabs from row r0 on, by two bulk copies.
template <class FG>
__device__ __forceinline__ void fu_tables(unsigned char *raw, const ulonglong2 *colt,
                                          const ulonglong2 *rowt, int prime, int r0, u64 *bar) {
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_expect_tx(bar, FG::TW_BYTES);
    bulk_g2s(raw, colt + ((size_t)prime << FG::LOGA), FG::N1 * 16, bar);
    bulk_g2s(raw + FG::N1 * 16,
             rowt + (((size_t)prime << FG::LOGA) + r0 << FG::LOGB), FG::PTS * 16, bar);
  }
}

// Column pass of the eight points v (column g of the CTA, thread t of the column), then the
// points to their rows' owners: CTA y / RC, row y % RC of its tile `ext`.
template <class FG, class SYNC>
__device__ __forceinline__ void fu_columns(u64 *v, u64 *colbuf, const ulonglong2 *twc, u64 m,
                                           int cls, int t, int g, int rank, const u64 *ext,
                                           SYNC sync) {
  if (cls == CLS_FAST)
    core::col_fwd<FG::LOGA, 3, FG::CC, CLS_FAST, 0>(v, colbuf, twc, m, t, g, sync);
  else if (cls == CLS_MID)
    core::col_fwd<FG::LOGA, 3, FG::CC, CLS_MID, 0>(v, colbuf, twc, m, t, g, sync);
  else
    core::col_fwd<FG::LOGA, 3, FG::CC, CLS_EXACT, 0>(v, colbuf, twc, m, t, g, sync);
  // the last round leaves rows 8t .. 8t + 7, of one owner
  const int y0 = 8 * t;
  const uint32_t base =
      cluster_map(ext, y0 / FG::RC) +
      8 * ((y0 % FG::RC) * FG::RP + core::row_pos(rank * FG::CC + g));
#pragma unroll
  for (int r = 0; r < 8; ++r) cluster_st(base + 8 * r * FG::RP, v[r]);
}

// Row pass of row `row` of the tile ext, in place: lazy result (canonical if canon).
template <class FG>
__device__ __forceinline__ void fu_row(u64 *s, const ulonglong2 *tw, const ModInfo &mi, u64 m,
                                       int cls, int t, bool canon) {
  u64 v[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) v[u] = s[core::row_pos((u << FG::SB::LOGT) + t)];
  row_fwd_cls<FG>(v, s, tw, m, t, cls);
  if (canon) {
    const u64 mu = mi.mu;
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = fwd_canon(v[r], m, mu, cls);
  }
  __syncwarp();
  core::put_row<typename FG::SB>(s, v, t);
}

template <int LOGN>
__global__ void __launch_bounds__(FuGeo<LOGN>::NT)
    k_fu_inv(KArgs a, JobSet js, WsOff wo, int which) {
  using FG = FuGeo<LOGN>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  cluster_arrive();
  const ulonglong2 *twc = reinterpret_cast<const ulonglong2 *>(raw), *twr = twc + FG::N1;
  u64 *tile = reinterpret_cast<u64 *>(raw + FG::TW_BYTES), *colbuf = tile + FG::ROWW;
  const JobPtr &jp = js.j[blockIdx.z];
  const InttSet is = intt_set(a, jp, wo, which);
  const int rank = blockIdx.x, inner = which == 0 ? a.nq : a.np;
  const int o = blockIdx.y / inner, ii = blockIdx.y - o * inner, prime = is.prime_base + ii;
  // the mirrored rows' slabs (see ks_ntt.cuh)
  fu_tables<FG>(raw, a.tab.twc_i, a.tab.twr_f, prime, (kFuC - 1 - rank) * FG::RC, &twbar);
  const ModInfo &mi = a.tab.mod[prime];
  const u64 m = mi.m, mu = mi.mu;
  const int cls = mod_class(m);
  const ulonglong2 sc = is.scale[ii];
  // an input in host memory: see inv_row_body
  const bool host_in = which == 0 && jp.dsrc, ahead = host_in && jp.ahead;
  if (!ahead) pdl_wait();
  const int row = threadIdx.x / FG::T2, t2 = threadIdx.x % FG::T2, w0 = row / FG::WR * FG::WR;
  const size_t off = (size_t)(rank * FG::RC + w0) << FG::LOGB;
  const u64 *src = (host_in ? jp.dsrc + ((size_t)ii << LOGN)
                            : is.src + ((size_t)(o * is.src_outer + ii) << LOGN)) +
                   off;
  u64 *ws = tile + w0 * FG::RP;
  input_rows<FG>(ws, src, host_in ? const_cast<u64 *>(jp.d) + ((size_t)ii << LOGN) + off : nullptr,
                 (a.nq << LOGN) > kPacedWords);
  __syncthreads();  // the warp's rows, and the barrier's initialisation
  tw_ready<true>(&twbar, a.tab.err);
  u64 v[8];
  u64 *s = tile + row * FG::RP;
  core::get_row<typename FG::SB>(v, s, t2);
  row_inv_cls<FG>(v, s, twr + (size_t)(FG::RC - 1 - row) * FG::N2, m, t2, cls);
  cluster_wait();  // every CTA of the cluster runs
  const int y = rank * FG::RC + row;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int x = (u << FG::SB::LOGT) + t2;
    cluster_st(cluster_map(colbuf, x / FG::CC) + 8 * (core::col_pos<3>(y) * FG::CC + x % FG::CC),
               inv_between(v[u], m, mu, cls));
  }
  cluster_arrive();
  cluster_wait();
  const int g = threadIdx.x % FG::CC, t = threadIdx.x / FG::CC;
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = colbuf[core::col_pos<3>(FG::CL::point(t, r)) * FG::CC + g];
  auto sync = [] { __syncthreads(); };
  if (cls == CLS_FAST)
    core::col_inv<FG::LOGA, 3, FG::CC, CLS_FAST, FG::KL>(v, colbuf, twc, m, t, g, sync);
  else if (cls == CLS_MID)
    core::col_inv<FG::LOGA, 3, FG::CC, CLS_MID, FG::KL>(v, colbuf, twc, m, t, g, sync);
  else
    core::col_inv<FG::LOGA, 3, FG::CC, CLS_EXACT, FG::KL>(v, colbuf, twc, m, t, g, sync);
  u64 *d = is.dst + ((size_t)(o * is.dst_outer + ii) << LOGN) + rank * FG::CC + g;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    d[(size_t)(u * FG::T1 + t) << FG::LOGB] = csub(shoup(v[u], sc.x, sc.y, m), m);
  if (ahead) pdl_wait();
  pdl_trigger();
}

// All digits of one target limb. Groups of NT threads take the digits in turn; the digits'
// row tiles stay in shared memory until the multiply.
template <int LOGN>
__global__ void __launch_bounds__(kFuThreads, 1) k_fu_up(KArgs a, JobSet js, WsOff wo) {
  using FG = FuGeo<LOGN>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  cluster_arrive();
  const ulonglong2 *twc = reinterpret_cast<const ulonglong2 *>(raw), *twr = twc + FG::N1;
  u64 *ext = reinterpret_cast<u64 *>(raw + FG::TW_BYTES), *colbufs = ext + a.beta * FG::ROWW;
  const JobPtr &jp = js.j[blockIdx.z];
  const int rank = blockIdx.x, tgt = gridDim.y - 1 - blockIdx.y;  // P-limb targets first
  const int grp = threadIdx.x / FG::NT, ngrp = blockDim.x / FG::NT, tl = threadIdx.x % FG::NT;
  u64 *colbuf = colbufs + grp * FG::COLW;
  const int od = tgt < a.nq ? tgt / a.alpha : -1;  // the target's own digit
  const int off0 = rank * FG::PTS;                 // the CTA's rows
  const u64 *evk = jp.evk + ((size_t)(tgt < a.nq ? tgt : a.epb + (tgt - a.nq)) << LOGN) + off0;
  fu_tables<FG>(raw, a.tab.twc_f, a.tab.twr_f, tgt, rank * FG::RC, &twbar);
  for (int k = threadIdx.x; k < 2 * a.beta; k += blockDim.x)
    prefetch_l2(evk + ((size_t)(k * a.eqp) << LOGN), FG::PTS * 8);
  const ModInfo &mi = a.tab.mod[tgt];
  const u64 m = mi.m;
  const int cls = mod_class(m);
  const bool lazy = cls == CLS_FAST && __umul64hi(kFwdLazy * a.beta, m) == 0;
  const int g = tl % FG::CC, t = tl / FG::CC;               // column pass
  const int row = tl / FG::T2, t2 = tl % FG::T2, w0 = row / FG::WR * FG::WR;  // row pass
  auto gsync = [&] {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(FG::NT) : "memory");
  };
  pdl_wait();
  __syncthreads();  // the table barrier's initialisation
  cluster_wait();   // every CTA of the cluster runs
  tw_ready<true>(&twbar, a.tab.err);
  for (int j = grp; j < a.beta; j += ngrp) {
    if (j == od) {
      own_rows<FG>(ext + j * FG::ROWW + w0 * FG::RP,
                   jp.d + ((size_t)tgt << LOGN) + off0 + (w0 << FG::LOGB), mi, lazy);
      continue;
    }
    u64 v[8];
    bconv_points<PRO_UP, LOGN>(v, a, tgt, j, jp.ws + wo.v + rank * FG::CC + g, t, cls);
    fu_columns<FG>(v, colbuf, twc, m, cls, t, g, rank, ext + j * FG::ROWW, gsync);
    gsync();  // colbuf is free for the group's next digit
  }
  cluster_arrive();
  cluster_wait();
  for (int j = grp; j < a.beta; j += ngrp)
    if (j != od) fu_row<FG>(ext + j * FG::ROWW + row * FG::RP, twr + row * FG::N2, mi, m, cls, t2,
                            !lazy);
  mac_tile<FG::LOGB, FG::RP, true>(mi, ext, FG::ROWW, a.beta, FG::PTS, evk, (size_t)a.eqp << LOGN,
                             jp.ws + wo.acc + ((size_t)tgt << LOGN) + off0,
                             (size_t)a.qp << LOGN, true, cls, [] { __syncthreads(); });
  pdl_trigger();
}

template <int LOGN>
__global__ void __launch_bounds__(FuGeo<LOGN>::NT)
    k_fu_down(KArgs a, JobSet js, WsOff wo) {
  using FG = FuGeo<LOGN>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ u64 twbar;
  cluster_arrive();
  const JobPtr &jp = js.j[blockIdx.z];
  if (jp.dsrc) pdl_trigger();  // host-buffer operation: see k_fwd_row_moddown
  const ulonglong2 *twc = reinterpret_cast<const ulonglong2 *>(raw), *twr = twc + FG::N1;
  u64 *ext = reinterpret_cast<u64 *>(raw + FG::TW_BYTES), *colbuf = ext + FG::ROWW;
  const int rank = blockIdx.x, i = blockIdx.y >> 1, c = blockIdx.y & 1;
  fu_tables<FG>(raw, a.tab.twc_f, a.tab.twr_f, i, rank * FG::RC, &twbar);
  const u64 m = a.tab.mod[i].m;
  const ulonglong2 pv = a.tab.pinv[i];
  const int cls = mod_class(m);
  const int g = threadIdx.x % FG::CC, t = threadIdx.x / FG::CC;
  const int row = threadIdx.x / FG::T2, t2 = threadIdx.x % FG::T2, w0 = row / FG::WR * FG::WR;
  const size_t woff = (size_t)(rank * FG::RC + w0) << FG::LOGB;  // the warp's rows
  const u64 *ac = jp.ws + wo.acc + ((size_t)(c * a.qp + i) << LOGN) + woff;
  auto sync = [] { __syncthreads(); };
  pdl_wait();
  if ((threadIdx.x & 31) == 0) prefetch_l2(ac, FG::WR * FG::N2 * 8);
  u64 v[8];
  bconv_points<PRO_DOWN, LOGN>(v, a, i, c, jp.ws + wo.vp + rank * FG::CC + g, t, cls);
  __syncthreads();  // the table barrier's initialisation
  cluster_wait();   // every CTA of the cluster runs
  tw_ready<true>(&twbar, a.tab.err);
  fu_columns<FG>(v, colbuf, twc, m, cls, t, g, rank, ext, sync);
  cluster_arrive();
  cluster_wait();
  fu_row<FG>(ext + row * FG::RP, twr + row * FG::N2, a.tab.mod[i], m, cls, t2, false);
  __syncwarp();
  const u64 *ws = ext + w0 * FG::RP;
  scale_rows<FG>(jp, c, ws, ac, ((size_t)(c * a.nq + i) << LOGN) + woff, pv, m, cls, false);
  pdl_trigger();
}

// ---------------------------------------------------------------------------
// Launch `kernel` with clusters of kFuC CTAs along x, chained like launch_pdl.
template <class... KT, class... AT>
inline cudaError_t launch_cluster(void (*kernel)(KT...), dim3 grid, int threads, size_t smem,
                                  cudaStream_t s, AT &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = kFuC;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<AT &&>(args)...);
}

template <int LOGN>
struct FusedFns {
  using FG = FuGeo<LOGN>;
  static constexpr int kSmemMax = 227 * 1024 - 1024;
  // groups of threads that take the digits in turn
  static int groups(int beta) { return std::max(1, std::min(beta, kFuThreads / FG::NT)); }
  static bool fits(int beta) { return FG::smem_up(beta, groups(beta)) <= kSmemMax; }
  static cudaError_t prepare_inv() { return smem_attr(k_fu_inv<LOGN>, FG::smem_inv()); }
  static cudaError_t inv(const ks_context *c, const JobSet &js, const WsOff &wo, int which,
                         cudaStream_t s) {
    return launch_cluster(k_fu_inv<LOGN>, dim3(kFuC, which == 0 ? c->nq : 2 * c->np, js.n),
                          FG::NT, FG::smem_inv(), s, args_of(c), js, wo, which);
  }
  static cudaError_t prepare() {
    cudaError_t e;
    if ((e = prepare_inv())) return e;
    if ((e = smem_attr(k_fu_down<LOGN>, FG::smem_inv()))) return e;
    return smem_attr(k_fu_up<LOGN>, kSmemMax);
  }
  static cudaError_t up(const ks_context *c, const JobSet &js, const WsOff &wo,
                        cudaStream_t s) {
    const int G = groups(c->beta);
    return launch_cluster(k_fu_up<LOGN>, dim3(kFuC, c->qp, js.n), G * FG::NT,
                          FG::smem_up(c->beta, G), s, args_of(c), js, wo);
  }
  static cudaError_t down(const ks_context *c, const JobSet &js, const WsOff &wo,
                          cudaStream_t s) {
    return launch_cluster(k_fu_down<LOGN>, dim3(kFuC, 2 * c->nq, js.n), FG::NT, FG::smem_inv(), s,
                          args_of(c), js, wo);
  }
  static const FusedTable &table() {
    static const FusedTable t = {&prepare, &fits, &up, &down, &inv};
    return t;
  }
  // only the inverse transform
  static bool no_fit(int) { return false; }
  static const FusedTable &table_inv() {
    static const FusedTable t = {&prepare_inv, &no_fit, nullptr, nullptr, &inv};
    return t;
  }
};

}  // namespace kern
}  // namespace ks
