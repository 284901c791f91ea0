// KeySwitch kernel templates for sm_103a, specialised per N = 2^LOGN: what every unit shares
// (arguments, task decoding, launches), the kernels of the single-pass sizes (N <= 2^11) and
// the stage bodies of the persistent batch (ks_persist.cu). The two-pass sizes' own kernels
// are in ks_rows.cuh, ks_tc.cu and ks_fused.cuh.
//
// Negacyclic NTT / iNTT (the two-pass sizes: column pass, row pass) with the fast basis
// conversions fused into the first forward pass and the key multiply or the
// ModDown scaling fused into the last one (Sec. II-A, Fig. 1). Twiddles of a tile
// are staged into shared memory once per CTA and reused for every polynomial the
// CTA transforms (all digits of a target limb; both accumulators in ModDown).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "ks_arith.cuh"
#include "ks_internal.h"
#include "ks_ntt.cuh"

namespace ks {
namespace kern {

enum { PRO_LOAD = 0, PRO_UP = 1, PRO_DOWN = 2 };

struct KArgs {
  Tables tab;
  int N, nq, np, qp, alpha, beta;
  int run_up, run_down;
  int eqp, epb;  // key layout (see ks_context)
  int tc_ap, tc_tplog;  // tensor-core basis conversion (see ks_context)
  int early;            // let the next kernel launch at this one's start (early_rule)
};

// Word offset of evk[j][c][limb t] (t in the context's Q u P numbering).
__host__ __device__ __forceinline__ size_t evk_off(const KArgs &a, int j, int c, int t) {
  const int tt = t < a.nq ? t : a.epb + (t - a.nq);
  return ((size_t)(j * 2 + c) * a.eqp + tt) * (size_t)a.N;
}

// The epilogue store of an output word: out = r, or r + addend (mod m).
__device__ __forceinline__ u64 out_word(const JobPtr &jp, int c, size_t idx, u64 r, u64 m) {
  if ((jp.addmask >> c) & 1) r = addmod(r, jp.add[idx], m);
  return r;
}

inline KArgs make_args(const ks_context *c) {
  KArgs a;
  a.tab = c->tab;
  a.N = c->N;
  a.nq = c->nq;
  a.np = c->np;
  a.qp = c->qp;
  a.alpha = c->alpha;
  a.beta = c->beta;
  a.run_up = c->run_up;
  a.run_down = c->run_down;
  a.eqp = c->eqp;
  a.epb = c->epb;
  a.tc_ap = c->tc_ap;
  a.tc_tplog = c->tc_tplog;
  a.early = 0;
  return a;
}

// Work item y of a task descriptor (see Tasks in ks_internal.h).
__host__ __device__ __forceinline__ uint32_t decode(const KArgs &a, const Tasks &tk, int y) {
  if (tk.mode == TASK_UP) {
    for (int j = tk.j0; j < tk.j1; ++j) {
      const int lo = j * a.alpha, hi = lo + a.alpha < a.nq ? lo + a.alpha : a.nq;
      const int ovl = lo > tk.t0 ? lo : tk.t0;
      const int ovh = hi < tk.t1 ? hi : tk.t1;
      const int ov = ovh - ovl > 0 ? ovh - ovl : 0;
      const int cnt = (tk.t1 - tk.t0) - ov;
      if (y < cnt) {
        int t = tk.t0 + y;
        if (ov > 0 && t >= ovl) t += ov;
        return pack_task(t, j, j * tk.sm.sj + t * tk.sm.st + tk.sm.base);
      }
      y -= cnt;
    }
    return 0;
  }
  if (tk.mode == TASK_TARGET) return pack_task(tk.t0 + y, 0, 0);
  if (tk.mode == TASK_DOWN) {
    const int n = tk.i1 - tk.i0, c = y / n, i = tk.i0 + y % n;
    return pack_task(i, c, c * tk.span + i - tk.ibase);
  }
  if (tk.mode == TASK_DOWN1) {
    const int i = tk.i0 + y;
    return pack_task(i, 0, i - tk.ibase);
  }
  return pack_task(y % a.qp, 0, y);
}

inline int count_tasks(const ks_context *c, const Tasks &tk) {
  switch (tk.mode) {
    case TASK_UP: {
      int n = 0;
      for (int j = tk.j0; j < tk.j1; ++j) {
        const int lo = j * c->alpha, hi = std::min(lo + c->alpha, c->nq);
        const int ov = std::max(0, std::min(hi, tk.t1) - std::max(lo, tk.t0));
        n += (tk.t1 - tk.t0) - ov;
      }
      return n;
    }
    case TASK_TARGET: return tk.t1 - tk.t0;
    case TASK_DOWN: return 2 * (tk.i1 - tk.i0);
    case TASK_DOWN1: return tk.i1 - tk.i0;
    default: return tk.n;
  }
}

// ---------------------------------------------------------------------------
// Tile movement. Rows r0..r0+G-1 of a limb are contiguous; columns c0..c0+G-1
// are G contiguous words in each of the N1 rows. 16-byte vector accesses,
// plain (coherent) loads: some kernels transform a buffer in place.

template <class GT>
__device__ __forceinline__ void load_rows(u64 *s, const u64 *src, int r0) {
  constexpr int TILE = GT::TILE, LOGB = GT::LOGB, P = GT::PR;
  const ulonglong2 *s2 = reinterpret_cast<const ulonglong2 *>(src + ((size_t)r0 << LOGB));
#pragma unroll
  for (int it = 0; it < (TILE / 2 + GT::NT - 1) / GT::NT; ++it) {
    const int e2 = threadIdx.x + it * GT::NT;
    if ((TILE / 2) % GT::NT != 0 && e2 >= TILE / 2) break;
    const ulonglong2 val = s2[e2];
    const int e = 2 * e2, g = e >> LOGB, x = e & ((1 << LOGB) - 1);
    s[x * P + g] = val.x;
    s[(x + 1) * P + g] = val.y;
  }
}

// load_rows that also writes the loaded words to `copy` (same layout): the input
// read from host memory leaves its device copy on the way.
template <class GT>
__device__ __forceinline__ void load_rows_copy(u64 *s, const u64 *src, u64 *copy, int r0) {
  constexpr int TILE = GT::TILE, LOGB = GT::LOGB, P = GT::PR;
  const ulonglong2 *s2 = reinterpret_cast<const ulonglong2 *>(src + ((size_t)r0 << LOGB));
  ulonglong2 *c2 = reinterpret_cast<ulonglong2 *>(copy + ((size_t)r0 << LOGB));
#pragma unroll
  for (int it = 0; it < (TILE / 2 + GT::NT - 1) / GT::NT; ++it) {
    const int e2 = threadIdx.x + it * GT::NT;
    if ((TILE / 2) % GT::NT != 0 && e2 >= TILE / 2) break;
    const ulonglong2 val = s2[e2];
    c2[e2] = val;
    const int e = 2 * e2, g = e >> LOGB, x = e & ((1 << LOGB) - 1);
    s[x * P + g] = val.x;
    s[(x + 1) * P + g] = val.y;
  }
}

template <class GT>
__device__ __forceinline__ void store_rows(u64 *dst, const u64 *s, int r0, u64 m, u64 mu) {
  // lazy values -> canonical
  constexpr int TILE = GT::TILE, LOGB = GT::LOGB, P = GT::PR;
  ulonglong2 *d2 = reinterpret_cast<ulonglong2 *>(dst + ((size_t)r0 << LOGB));
#pragma unroll
  for (int it = 0; it < (TILE / 2 + GT::NT - 1) / GT::NT; ++it) {
    const int e2 = threadIdx.x + it * GT::NT;
    if ((TILE / 2) % GT::NT != 0 && e2 >= TILE / 2) break;
    const int e = 2 * e2, g = e >> LOGB, x = e & ((1 << LOGB) - 1);
    ulonglong2 val;
    val.x = reduce_full(s[x * P + g], m, mu);
    val.y = reduce_full(s[(x + 1) * P + g], m, mu);
    d2[e2] = val;
  }
}

template <class GT>
__device__ __forceinline__ void load_cols(u64 *s, const u64 *src, int c0) {
  constexpr int TILE = GT::N1 * GT::GC, LOGG = GT::LOGGC, P = GT::PC;
#pragma unroll
  for (int it = 0; it < (TILE / 2 + GT::NT - 1) / GT::NT; ++it) {
    const int e2 = threadIdx.x + it * GT::NT;
    if ((TILE / 2) % GT::NT != 0 && e2 >= TILE / 2) break;
    const int e = 2 * e2, y = e >> LOGG, g = e & ((1 << LOGG) - 1);
    const ulonglong2 val =
        *reinterpret_cast<const ulonglong2 *>(src + ((size_t)y << GT::LOGB) + c0 + g);
    s[y * P + g] = val.x;
    s[y * P + g + 1] = val.y;
  }
}

template <class GT>
__device__ __forceinline__ void store_cols(u64 *dst, const u64 *s, int c0) {
  constexpr int TILE = GT::N1 * GT::GC, LOGG = GT::LOGGC, P = GT::PC;
#pragma unroll
  for (int it = 0; it < (TILE / 2 + GT::NT - 1) / GT::NT; ++it) {
    const int e2 = threadIdx.x + it * GT::NT;
    if ((TILE / 2) % GT::NT != 0 && e2 >= TILE / 2) break;
    const int e = 2 * e2, y = e >> LOGG, g = e & ((1 << LOGG) - 1);
    ulonglong2 val;
    val.x = s[y * P + g];
    val.y = s[y * P + g + 1];
    *reinterpret_cast<ulonglong2 *>(dst + ((size_t)y << GT::LOGB) + c0 + g) = val;
  }
}

// Stage n twiddle pairs (a contiguous slab of the table) into shared memory with one
// TMA bulk copy: thread 0 arms the CTA's barrier `bar` and issues the copy, which then
// lands while the kernel waits for its predecessor and loads its data tile. Every thread
// calls tw_ready before the first round that reads the twiddles, after a barrier that
// follows stage_tw (so the barrier's initialisation is visible).
// TMA = false (the persistent kernel, whose CTAs run many tiles): every thread copies
// its share with ordinary loads instead, and tw_ready is a no-op (the barrier before
// the first round orders the stores).
template <class GT, bool TMA = true>
__device__ __forceinline__ void stage_tw(ulonglong2 *tws, const ulonglong2 *__restrict__ src,
                                         int n, u64 *bar) {
  if (TMA) {
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      mbar_expect_tx(bar, (unsigned)n * 16);
      bulk_g2s(tws, src, (unsigned)n * 16, bar);
    }
  } else {
    const u64 pol = l2_keep();
    for (int k = threadIdx.x; k < n; k += GT::NT) tws[k] = ldg_pol(src + k, pol);
  }
}
// The twiddles of a row tile: the table's slab, each row's entries at a pitch of N2 + 1 (two-pass
// sizes). With the rows at the table's own pitch the persistent batch's row stages met GR-way
// bank conflicts: 64-job batch 23.0 ms against 21.4.
template <class GT, bool TMA = true>
__device__ __forceinline__ void stage_row_slab(ulonglong2 *tws,
                                               const ulonglong2 *__restrict__ src, u64 *bar) {
  if (GT::LOGA == 0) {
    stage_tw<GT, TMA>(tws, src, GT::TWR, bar);
  } else if (TMA) {
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      mbar_expect_tx(bar, GT::TWR * 16);
      for (int g = 0; g < GT::GR; ++g)
        bulk_g2s(tws + g * (GT::N2 + 1), src + g * GT::N2, GT::N2 * 16, bar);
    }
  } else {
    const u64 pol = l2_keep();
    for (int k = threadIdx.x; k < GT::TWR; k += GT::NT)
      tws[k + (k >> GT::LOGB)] = ldg_pol(src + k, pol);
  }
}
// Wait for the twiddle slab; a wait that gives up records it in the context's error
// word (ks_sync_status then returns KS_ETIMEOUT) and carries on.
template <bool TMA = true>
__device__ __forceinline__ void tw_ready(u64 *bar, int *err) {
  if (TMA && !mbar_wait(bar, 0)) atomicExch(err, 1);
}

// Column-pass twiddles of a prime: the first N1 entries of its column table.
template <class GT>
__device__ __forceinline__ const ulonglong2 *col_table(const ulonglong2 *tab, int prime) {
  return tab + ((size_t)prime << GT::LOGA);
}
// Row-pass twiddle slab of (prime, row tile blk): N2 entries per row (a single pass: N-1).
template <class GT>
__device__ __forceinline__ const ulonglong2 *row_table(const ulonglong2 *tab, int prime,
                                                       int blk) {
  return tab + (size_t)prime * (GT::TWR / GT::GR) * GT::N1 + (size_t)blk * GT::TWR;
}

__device__ __forceinline__ void stage_consts(u64 *cst, const u64 *__restrict__ src, int n,
                                             int nt) {
  for (int k = threadIdx.x; k < n; k += nt) cst[k] = __ldg(src + k);
}

// Fast basis conversion into a tile: element -> REDC(sum_k src_k[gidx] * cst[k]),
// in runs of at most `run` terms per exact 128-bit sum. Output in [0, 2m).
// COL: column tile (element (y, g) = limb index y*N2 + base + g);
// otherwise row tile (element (x, g) = limb index (base + g)*N2 + x).
template <class GT, bool COL>
__device__ __forceinline__ void bconv_tile(u64 *s, const u64 *src, size_t N,
                                           int nsrc, const u64 *cst, int run, int base, u64 m,
                                           u64 minv) {
  constexpr int LOGG = COL ? GT::LOGGC : GT::LOGGR;
  constexpr int TILE = COL ? GT::N1 * GT::GC : GT::N2 * GT::GR;
  constexpr int P = COL ? GT::PC : GT::PR;
  constexpr int EPT = (TILE + GT::NT - 1) / GT::NT;
  constexpr int H = EPT >= 4 ? 4 : EPT;  // elements per batch (bounds live registers)
  const u64 m2 = 2 * m;
#pragma unroll 1
  for (int k0 = 0; k0 < EPT; k0 += H) {
    int gi[H];
    U128 acc[H];
    u64 z[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const int e = threadIdx.x + (k0 + k) * GT::NT;
      if (COL) {
        const int y = e >> LOGG, g = e & ((1 << LOGG) - 1);
        gi[k] = (y << GT::LOGB) + base + g;
      } else {
        const int g = e >> GT::LOGB, x = e & ((1 << GT::LOGB) - 1);
        gi[k] = ((base + g) << GT::LOGB) + x;
      }
      acc[k] = U128{0, 0};
      z[k] = 0;
    }
    int cnt = 0;
    // loads of source limb i+1 are issued before the products of limb i
    u64 x[H];
#pragma unroll
    for (int k = 0; k < H; ++k)
      x[k] = (TILE % GT::NT == 0 || threadIdx.x + (k0 + k) * GT::NT < TILE) ? src[gi[k]] : 0;
    for (int i = 0; i < nsrc; ++i) {
      const u64 c = cst[i];
      u64 xn[H];
      if (i + 1 < nsrc) {
        const u64 *sn = src + (size_t)(i + 1) * N;
#pragma unroll
        for (int k = 0; k < H; ++k)
          xn[k] = (TILE % GT::NT == 0 || threadIdx.x + (k0 + k) * GT::NT < TILE) ? sn[gi[k]] : 0;
      }
#pragma unroll
      for (int k = 0; k < H; ++k) mac128(acc[k], x[k], c);
      if (++cnt == run || i == nsrc - 1) {
#pragma unroll
        for (int k = 0; k < H; ++k) {
          const u64 zz = z[k] + redc(acc[k], m, minv);
          z[k] = zz >= m2 ? zz - m2 : zz;
          acc[k] = U128{0, 0};
        }
        cnt = 0;
      }
      if (i + 1 < nsrc) {
#pragma unroll
        for (int k = 0; k < H; ++k) x[k] = xn[k];
      }
    }
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const int e = threadIdx.x + (k0 + k) * GT::NT;
      if (TILE % GT::NT != 0 && e >= TILE) break;
      const int sidx = COL ? (e >> LOGG) * P + (e & ((1 << LOGG) - 1))
                           : (e & ((1 << GT::LOGB) - 1)) * P + (e >> GT::LOGB);
      s[sidx] = z[k];
    }
  }
}

// Produce the tile of task w: BConv (ModUp: digit j onto limb t, Montgomery-scaled
// by constants carrying 2^128; ModDown: P-limbs of polynomial c onto q_i) or a
// plain load of buf[slot].
template <class GT, int PRO, bool COL>
__device__ __forceinline__ void produce(const KArgs &a, u64 *sm, u64 *cst, uint32_t w,
                                        const u64 *__restrict__ v, const u64 *buf, int base) {
  const int t = task_limb(w);
  const size_t N = a.N;
  if (PRO == PRO_LOAD) {
    const u64 *b = buf + (size_t)task_slot(w) * N;
    if (COL)
      load_cols<GT>(sm, b, base);
    else
      load_rows<GT>(sm, b, base);
  } else if (PRO == PRO_UP) {
    const int j = task_dig(w);
    const int i0 = j * a.alpha;
    const int ns = min(a.nq, i0 + a.alpha) - i0;
    stage_consts(cst, a.tab.cup + ((size_t)j * a.qp + t) * a.alpha, ns, GT::NT);
    __syncthreads();
    const ModInfo mi = a.tab.mod[t];
    bconv_tile<GT, COL>(sm, v + (size_t)i0 * N, N, ns, cst, a.run_up, base, mi.m, mi.minv);
  } else {
    const int c = task_dig(w);
    stage_consts(cst, a.tab.cdown + (size_t)t * a.alpha, a.np, GT::NT);
    __syncthreads();
    const ModInfo mi = a.tab.mod[t];
    bconv_tile<GT, COL>(sm, v + (size_t)c * a.np * N, N, a.np, cst, a.run_down, base, mi.m,
                        mi.minv);
  }
}

// Shared-memory layout of the kernels: twiddles first (16-byte aligned), then
// the tile.
template <class GT, bool COL>
__device__ __forceinline__ u64 *tile_ptr(unsigned char *raw) {
  return reinterpret_cast<u64 *>(raw + (COL ? GT::TWC : GT::TWS) * 16);
}

// ---------------------------------------------------------------------------
// Kernels. grid (tiles, work items, jobs); the job's pointers are js.j[blockIdx.z].

// Minimum resident blocks for a target of `threads` threads per SM (register cap).
__host__ __device__ constexpr int min_blocks(int nt, int threads) {
  return threads / nt > 0 ? threads / nt : 1;
}

// iNTT limb set `which`: 0 = the L+1 input limbs (d -> v), 1 = the P-limbs of both
// accumulators (acc -> vp). Returns (src, src_outer, dst, dst_outer, outer, prime_base,
// scale) for the current job.
struct InttSet {
  const u64 *src;
  u64 *dst;
  int src_outer, dst_outer, outer, prime_base;
  const ulonglong2 *scale;
};
__device__ __forceinline__ InttSet intt_set(const KArgs &a, const JobPtr &jp, const WsOff &o,
                                            int which) {
  InttSet r;
  if (which == 0) {
    r.src = jp.d;
    r.dst = jp.ws + o.v;
    r.src_outer = r.dst_outer = 0;
    r.outer = 1;
    r.prime_base = 0;
    r.scale = a.tab.iscale_q;
  } else {
    r.src = jp.ws + o.acc + (size_t)a.nq * a.N;
    r.dst = jp.ws + o.vp;
    r.src_outer = a.qp;
    r.dst_outer = a.np;
    r.outer = 2;
    r.prime_base = a.nq;
    r.scale = a.tab.iscale_p;
  }
  return r;
}

// Inverse NTT, row pass (global stages logN-1 .. logN1) of limb `by`: all `outer`
// polynomials in one CTA (shared twiddles), or only polynomial `only_o` when it is
// >= 0. With a single pass (N1 == 1) it also applies the per-limb scale (canonical
// output).
template <int LOGN, int RL, bool TMA = true>
__device__ __forceinline__ void inv_row_body(const KArgs &a, const JobPtr &jp, const WsOff &wo,
                                             int which, int bx, int by, unsigned char *raw,
                                             int only_o = -1) {
  using GT = GeoT<LOGN, RL, 1>;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *sm = tile_ptr<GT, false>(raw);
  const InttSet is = intt_set(a, jp, wo, which);
  const int ii = by, prime = is.prime_base + ii, blk = bx;
  const int r0 = blk * GT::GR;
  const u64 m = a.tab.mod[prime].m, mu = a.tab.mod[prime].mu;
  const size_t N = a.N;
  // inverse twiddles: the forward slab of the mirrored row tile (see ks_ntt.cuh)
  __shared__ u64 twbar;
  stage_row_slab<GT, TMA>(tws, row_table<GT>(a.tab.twr_f, prime, GT::N1 / GT::GR - 1 - blk),
                          &twbar);
  // Reading the input from host memory (`dsrc`), this pass writes only v and the device
  // copy of d, which no kernel of the previous operation on the stream reads once its
  // last kernel runs. Where that operation does not write the input either (`ahead`), it
  // starts without waiting, so its host reads overlap that kernel's host writes, and waits
  // for it at the end (keeping the chain's order for what follows).
  const bool ahead = which == 0 && jp.dsrc && jp.ahead;
  if (!ahead) pdl_wait();
  const ulonglong2 sc = is.scale[ii];
  const int o0 = only_o < 0 ? 0 : only_o, o1 = only_o < 0 ? is.outer : only_o + 1;
  for (int o = o0; o < o1; ++o) {
    if (which == 0 && jp.dsrc)
      load_rows_copy<GT>(sm, jp.dsrc + (size_t)ii * N, const_cast<u64 *>(jp.d) + (size_t)ii * N,
                         r0);
    else
      load_rows<GT>(sm, is.src + ((size_t)o * is.src_outer + ii) * N, r0);
    __syncthreads();
    tw_ready<TMA>(&twbar, a.tab.err);
    tile_inv<GT::LOGB, GT::LOGGR, GT::PR, GT::NT, true, RL>(sm, tws, m);
    u64 *d = is.dst + ((size_t)o * is.dst_outer + ii) * N;
    if (GT::LOGA == 0) {
#pragma unroll
      for (int k = 0; k < GT::EPT; ++k) {
        const int e = threadIdx.x + k * GT::NT;
        if (GT::TILE % GT::NT != 0 && e >= GT::TILE) break;
        d[e] = csub(shoup(sm[e], sc.x, sc.y, m), m);
      }
    } else {
      store_rows<GT>(d, sm, r0, m, mu);
    }
    __syncthreads();
  }
  if (ahead) pdl_wait();
}

// Grid row of an inverse-NTT launch: the limb, and with `split` the polynomial too
// (blockIdx.y = o * limbs + limb), so that the two accumulator polynomials of the
// P-limbs run in separate CTAs when one CTA per limb would leave SMs idle.
__device__ __forceinline__ int inv_grid_row(const KArgs &a, int which, int split, int &only_o) {
  int by = blockIdx.y;
  only_o = -1;
  if (split) {
    const int inner = which == 0 ? a.nq : a.np;
    only_o = by / inner;
    by -= only_o * inner;
  }
  return by;
}

template <int LOGN, int RL>
__global__ void __launch_bounds__(GeoT<LOGN, RL, 1>::NT)
    k_inv_row(KArgs a, JobSet js, WsOff wo, int which, int split) {
  extern __shared__ __align__(16) unsigned char raw[];
  int only_o;
  const int by = inv_grid_row(a, which, split, only_o);
  inv_row_body<LOGN, RL>(a, js.j[blockIdx.z], wo, which, blockIdx.x, by, raw, only_o);
  pdl_trigger();  // the next kernel may launch once every CTA is here
}

// Inverse NTT, column pass (global stages logN1-1 .. 0), in place, then the per-limb scale.
template <int LOGN, int RL, bool TMA = true>
__device__ __forceinline__ void inv_col_body(const KArgs &a, const JobPtr &jp, const WsOff &wo,
                                             int which, int bx, int by, unsigned char *raw) {
  using GT = GeoT<LOGN, RL, 0>;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *sm = tile_ptr<GT, true>(raw);
  const InttSet is = intt_set(a, jp, wo, which);
  const int ii = by, prime = is.prime_base + ii;
  const int c0 = bx * GT::GC;
  const u64 m = a.tab.mod[prime].m;
  __shared__ u64 twbar;
  stage_tw<GT, TMA>(tws, col_table<GT>(a.tab.twc_i, prime), GT::TWC, &twbar);
  pdl_wait();
  const ulonglong2 sc = is.scale[ii];
  for (int o = 0; o < is.outer; ++o) {
    u64 *d = is.dst + ((size_t)o * is.dst_outer + ii) * (size_t)a.N;
    load_cols<GT>(sm, d, c0);
    __syncthreads();
    tw_ready<TMA>(&twbar, a.tab.err);
    tile_inv<GT::LOGA, GT::LOGGC, GT::PC, GT::NT, false, RL>(sm, tws, m);
    constexpr int TILE = GT::N1 * GT::GC;
#pragma unroll
    for (int k = 0; k < (TILE + GT::NT - 1) / GT::NT; ++k) {
      const int e = threadIdx.x + k * GT::NT;
      if (TILE % GT::NT != 0 && e >= TILE) break;
      const int y = e >> GT::LOGGC, g = e & (GT::GC - 1);
      sm[y * GT::PC + g] = csub(shoup(sm[y * GT::PC + g], sc.x, sc.y, m), m);
    }
    __syncthreads();
    store_cols<GT>(d, sm, c0);
    __syncthreads();
  }
}

// Buffers of a forward pass for job jp: the BConv sources and the output buffer.
template <int PRO>
__device__ __forceinline__ void fwd_bufs(const JobPtr &jp, const WsOff &wo, int buf,
                                         const u64 *&src, u64 *&dst) {
  if (PRO == PRO_UP) {
    src = jp.ws + wo.v;
    dst = jp.ws + wo.tmp;
  } else if (PRO == PRO_DOWN) {
    src = jp.ws + wo.vp;
    dst = jp.ws + wo.tmp2;
  } else {
    src = nullptr;
    dst = jp.ws + (buf == BUF_TMP ? wo.tmp : wo.tmp2);
  }
}

// Forward NTT, column pass (global stages 0 .. logN1-1) with a tile producer; the
// lazy result goes to the output buffer's slot.
template <int LOGN, int RL, int PRO, bool TMA = true>
__device__ __forceinline__ void fwd_col_body(const KArgs &a, const JobPtr &jp, const WsOff &wo,
                                             const Tasks &tk, int buf, int bx, int by,
                                             unsigned char *raw, u64 *cst) {
  using GT = GeoT<LOGN, RL, 0>;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *sm = tile_ptr<GT, true>(raw);
  const u64 *src;
  u64 *dst;
  fwd_bufs<PRO>(jp, wo, buf, src, dst);
  const uint32_t w = decode(a, tk, by);
  const int t = task_limb(w);
  const int c0 = bx * GT::GC;
  __shared__ u64 twbar;
  stage_tw<GT, TMA>(tws, col_table<GT>(a.tab.twc_f, t), GT::TWC, &twbar);
  pdl_wait();
  produce<GT, PRO, true>(a, sm, cst, w, src, dst, c0);
  __syncthreads();
  tw_ready<TMA>(&twbar, a.tab.err);
  tile_fwd<GT::LOGA, GT::LOGGC, GT::PC, GT::NT, false, RL>(sm, tws, a.tab.mod[t].m);
  store_cols<GT>(dst + (size_t)task_slot(w) * a.N, sm, c0);
}

// Plain forward row pass: canonical result back in place.
template <int LOGN, int RL>
__global__ void __launch_bounds__(GeoT<LOGN, RL, 1>::NT)
    k_fwd_row_store(KArgs a, JobSet js, WsOff wo, Tasks tk, int buf) {
  using GT = GeoT<LOGN, RL, 1>;
  constexpr bool TMA = true;
  extern __shared__ __align__(16) unsigned char raw[];
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *sm = tile_ptr<GT, false>(raw);
  const u64 *src;
  u64 *dst;
  fwd_bufs<PRO_LOAD>(js.j[blockIdx.z], wo, buf, src, dst);
  const uint32_t w = decode(a, tk, blockIdx.y);
  const int t = task_limb(w), blk = blockIdx.x, r0 = blk * GT::GR;
  const u64 m = a.tab.mod[t].m;
  __shared__ u64 twbar;
  stage_row_slab<GT, TMA>(tws, row_table<GT>(a.tab.twr_f, t, blk), &twbar);
  pdl_wait();
  u64 *b = dst + (size_t)task_slot(w) * a.N;
  load_rows<GT>(sm, b, r0);
  __syncthreads();
  tw_ready<TMA>(&twbar, a.tab.err);
  tile_fwd<GT::LOGB, GT::LOGGR, GT::PR, GT::NT, true, RL>(sm, tws, m);
  store_rows<GT>(b, sm, r0, m, a.tab.mod[t].mu);
  pdl_trigger();  // the next kernel may launch once every CTA is here
}

// ModUp row pass fused with the key multiply. One CTA = one row tile of one
// target limb t (TASK_TARGET), over digits j0..j1-1:
//   acc_c[t] (+)= sum_j ext_j[t] * evk[j][c][t],  c = 0, 1,
// with ext_j[t] = NTT(BConv_j)[t] (Montgomery-scaled) or, on digit j's own limbs,
// the input d_t (put in Montgomery form here), so that REDC of a sum of exact
// 128-bit products is the plain sum of products mod m. The row twiddles of (t, tile)
// are staged once.
//
// The products take ext as the forward pass leaves it (below kFwdLazy * m with the
// fast butterflies; the other classes: brought below m first),
// since REDC only needs its input below m 2^64. With at most four elements per
// thread the products of all digits are summed exactly in 128 bits and reduced once
// per output word (needs (bound of ext) * (digits) * m < 2^64, checked per CTA; the
// context guarantees digits * m < 2^64 for canonical ext); with more elements per
// thread (register budget) each product is reduced and the residues summed lazily.
template <int LOGN, int RL, int PRO, bool TMA = true>
__device__ __forceinline__ void keymult_body(const KArgs &a, const JobPtr &jp, const WsOff &wo,
                                             const Tasks &tk, int bx, int by,
                                             unsigned char *raw, u64 *cst) {
  using GT = GeoT<LOGN, RL, 1>;
  constexpr int EPT = GT::EPT;
  constexpr bool WIDE = EPT <= 4;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *sm = tile_ptr<GT, false>(raw);
  const u64 *v = jp.ws + wo.v, *tmp = jp.ws + wo.tmp;
  u64 *acc = jp.ws + wo.acc;
  const int t = task_limb(decode(a, tk, by));
  const ModInfo mi = a.tab.mod[t];
  const int blk = bx, r0 = blk * GT::GR;
  const size_t N = a.N;
  const size_t off0 = (size_t)r0 << GT::LOGB;  // the tile is contiguous from here
  // One thread asks the TMA unit to pull each digit's tiles (two evk tiles and the
  // ModUp intermediate, or d on the digit's own limbs) into L2 one digit ahead.
  constexpr unsigned TB = GT::TILE * 8;
  auto prefetch_digit = [&](int j) {
    if (threadIdx.x != 0 || j >= tk.j1) return;
    prefetch_l2(jp.evk + evk_off(a, j, 0, t) + off0, TB);
    prefetch_l2(jp.evk + evk_off(a, j, 1, t) + off0, TB);
    const int lo = j * a.alpha, hi = min(lo + a.alpha, a.nq);
    if (t >= lo && t < hi)
      prefetch_l2(jp.d + (size_t)t * N + off0, TB);
    else if (GT::LOGA != 0)
      prefetch_l2(tmp + (size_t)(j * tk.sm.sj + t * tk.sm.st + tk.sm.base) * N + off0, TB);
  };
  prefetch_digit(tk.j0);
  __shared__ u64 twbar;
  stage_row_slab<GT, TMA>(tws, row_table<GT>(a.tab.twr_f, t, blk), &twbar);
  pdl_wait();
  const u64 pol = l2_stream();
  const int cls = mod_class(mi.m);
  const bool fast = cls == CLS_FAST;
  // ext stays lazy when the exact digit sum of its products fits one REDC
  const int nd = tk.j1 - tk.j0;
  const bool lazy = fast && (unsigned __int128)(kFwdLazy * (WIDE ? nd : 1)) * mi.m <
                                (unsigned __int128)1 << 64;
  const u64 m2 = 2 * mi.m;
  auto ext_word = [&](u64 y) -> u64 {
    if (lazy) return y;
    return fwd_canon(y, mi.m, mi.mu, cls);
  };
  U128 w0[WIDE ? EPT : 1], w1[WIDE ? EPT : 1];  // exact digit sums (WIDE)
  u64 s0[WIDE ? 1 : EPT], s1[WIDE ? 1 : EPT];    // lazy residue sums in [0, 2m)
#pragma unroll
  for (int k = 0; k < (WIDE ? EPT : 1); ++k) w0[k] = w1[k] = U128{0, 0};
#pragma unroll
  for (int k = 0; k < (WIDE ? 1 : EPT); ++k) s0[k] = s1[k] = 0;
  auto mac_word = [&](int k, u64 y, const u64 *e0, const u64 *e1, int e) {
    if (WIDE) {
      mac128(w0[k], y, ldg_pol(e0 + e, pol));
      mac128(w1[k], y, ldg_pol(e1 + e, pol));
    } else {
      U128 p0 = {0, 0}, p1 = {0, 0};
      mac128(p0, y, ldg_pol(e0 + e, pol));
      mac128(p1, y, ldg_pol(e1 + e, pol));
      const u64 a0v = s0[k] + redc(p0, mi.m, mi.minv), a1v = s1[k] + redc(p1, mi.m, mi.minv);
      s0[k] = a0v >= m2 ? a0v - m2 : a0v;
      s1[k] = a1v >= m2 ? a1v - m2 : a1v;
    }
  };
  for (int j = tk.j0; j < tk.j1; ++j) {
    prefetch_digit(j + 1);
    const int lo = j * a.alpha, hi = min(lo + a.alpha, a.nq);
    const bool own = t >= lo && t < hi;
    const u64 *e0 = jp.evk + evk_off(a, j, 0, t) + off0;
    const u64 *e1 = jp.evk + evk_off(a, j, 1, t) + off0;
    if (own) {
      const u64 *dt = jp.d + (size_t)t * N + off0;
#pragma unroll
      for (int k = 0; k < EPT; ++k) {
        const int e = threadIdx.x + k * GT::NT;
        if (GT::TILE % GT::NT == 0 || e < GT::TILE) {
          u64 y = shoup(__ldg(dt + e), mi.r1, mi.r1s, mi.m);  // [0, 2m)
          if (!lazy) y = csub(y, mi.m);
          mac_word(k, y, e0, e1, e);
        }
      }
    } else {
      const int slot = j * tk.sm.sj + t * tk.sm.st + tk.sm.base;
      if (GT::LOGA == 0)
        produce<GT, PRO, false>(a, sm, cst, pack_task(t, j, slot), v, tmp, r0);
      else
        produce<GT, PRO_LOAD, false>(a, sm, cst, pack_task(t, j, slot), v, tmp, r0);
      __syncthreads();
      tw_ready<TMA>(&twbar, a.tab.err);
      tile_fwd<GT::LOGB, GT::LOGGR, GT::PR, GT::NT, true, RL>(sm, tws, mi.m);
#pragma unroll
      for (int k = 0; k < EPT; ++k) {
        const int e = threadIdx.x + k * GT::NT;
        if (GT::TILE % GT::NT == 0 || e < GT::TILE) {
          const int g = e >> GT::LOGB, x = e & (GT::N2 - 1);
          mac_word(k, ext_word(sm[x * GT::PR + g]), e0, e1, e);
        }
      }
      __syncthreads();
    }
  }
  u64 *a0 = acc + (size_t)t * N + off0;
  u64 *a1 = acc + ((size_t)a.qp + t) * N + off0;
#pragma unroll
  for (int k = 0; k < EPT; ++k) {
    const int e = threadIdx.x + k * GT::NT;
    if (GT::TILE % GT::NT != 0 && e >= GT::TILE) break;
    u64 r0v, r1v;
    if (WIDE) {
      r0v = csub(redc(w0[k], mi.m, mi.minv), mi.m);
      r1v = csub(redc(w1[k], mi.m, mi.minv), mi.m);
    } else {
      r0v = csub(s0[k], mi.m);
      r1v = csub(s1[k], mi.m);
    }
    if (!tk.first) {
      r0v = addmod(r0v, a0[e], mi.m);
      r1v = addmod(r1v, a1[e], mi.m);
    }
    a0[e] = r0v;
    a1[e] = r1v;
  }
}

// Shared memory of the pipelined key multiply: the row twiddles, two ext tiles (odd
// pitch) and two digits' key tiles (c = 0, 1, contiguous).
template <class GT>
struct KmSmem {
  static constexpr int TW = GT::TWS * 16;
  static constexpr int TILEW = GT::N2 * GT::PR;  // words of one pitched tile
  static constexpr int KEYW = 2 * GT::TILE;      // words of one digit's two key tiles
  static constexpr int BYTES = TW + 2 * TILEW * 8 + 2 * KEYW * 8;
};

// The key multiply of keymult_body for N >= 2^13 (persistent batch), software-pipelined over the digits:
// while digit j's ext tile is transformed and multiplied, the copies of digit j+1's
// tile (the ModUp intermediate, or d_t on the digit's own limbs: cp.async into the odd
// pitch) and of its two key tiles (TMA bulk copies on a barrier) are in flight into the
// other half of double buffers. Same arithmetic, same bounds and the same result as
// keymult_body.
template <int LOGN, int RL>
__device__ __forceinline__ void keymult_pipe_body(const KArgs &a, const JobPtr &jp,
                                                  const WsOff &wo, const Tasks &tk, int bx,
                                                  int by, unsigned char *raw) {
  using GT = GeoT<LOGN, RL, 1>;
  using SM = KmSmem<GT>;
  constexpr bool TMA = true;
  constexpr int EPT = GT::EPT, TILE = GT::TILE, NT = GT::NT;
  constexpr bool WIDE = EPT <= 4;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *tiles = reinterpret_cast<u64 *>(raw + SM::TW);
  u64 *keys = tiles + 2 * SM::TILEW;
  const u64 *tmp = jp.ws + wo.tmp;
  u64 *acc = jp.ws + wo.acc;
  const int t = task_limb(decode(a, tk, by));
  const ModInfo mi = a.tab.mod[t];
  const int blk = bx, r0 = blk * GT::GR;
  const size_t N = a.N;
  const size_t off0 = (size_t)r0 << GT::LOGB;  // the tile is contiguous from here
  auto own = [&](int j) {
    const int lo = j * a.alpha;
    return t >= lo && t < min(lo + a.alpha, a.nq);
  };
  // key tiles: two contiguous TILE-word tiles per digit, one TMA bulk copy each, on the
  // buffer's barrier (use k of buffer b completes phase k & 1)
  __shared__ u64 keybar[2];
  auto issue_keys = [&](int j, int b) {
    if (threadIdx.x != 0) return;
    const u64 *e0 = jp.evk + evk_off(a, j, 0, t) + off0;
    const u64 *e1 = jp.evk + evk_off(a, j, 1, t) + off0;
    u64 *k0 = keys + b * SM::KEYW;
    mbar_expect_tx(&keybar[b], 2 * TILE * 8);
    bulk_g2s(k0, e0, TILE * 8, &keybar[b]);
    bulk_g2s(k0 + TILE, e1, TILE * 8, &keybar[b]);
  };
  auto issue_tile = [&](int j, int b) {
    const u64 *src = own(j) ? jp.d + (size_t)t * N + off0
                            : tmp + (size_t)(j * tk.sm.sj + t * tk.sm.st + tk.sm.base) * N + off0;
    u64 *st = tiles + b * SM::TILEW;
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      const int w = threadIdx.x + k * NT;
      if (TILE % NT != 0 && w >= TILE) break;
      cp_async8(st + (w & (GT::N2 - 1)) * GT::PR + (w >> GT::LOGB), src + w);
    }
  };
  // the key tiles are inputs of the operation (no kernel of the chain writes them):
  // their first copies start before the wait for the previous kernel
  if (threadIdx.x == 0) {
    mbar_init(&keybar[0], 1);
    mbar_init(&keybar[1], 1);
  }
  issue_keys(tk.j0, 0);
  __shared__ u64 twbar;
  stage_row_slab<GT, TMA>(tws, row_table<GT>(a.tab.twr_f, t, blk), &twbar);
  pdl_wait();
  issue_tile(tk.j0, 0);
  cp_async_commit();
  const int cls = mod_class(mi.m);
  const bool fast = cls == CLS_FAST;
  const int nd = tk.j1 - tk.j0;
  const bool lazy = fast && (unsigned __int128)(kFwdLazy * (WIDE ? nd : 1)) * mi.m <
                                (unsigned __int128)1 << 64;
  const u64 m2 = 2 * mi.m;
  U128 w0[WIDE ? EPT : 1], w1[WIDE ? EPT : 1];  // exact digit sums (WIDE)
  u64 s0[WIDE ? 1 : EPT], s1[WIDE ? 1 : EPT];    // lazy residue sums in [0, 2m)
#pragma unroll
  for (int k = 0; k < (WIDE ? EPT : 1); ++k) w0[k] = w1[k] = U128{0, 0};
#pragma unroll
  for (int k = 0; k < (WIDE ? 1 : EPT); ++k) s0[k] = s1[k] = 0;
  for (int j = tk.j0; j < tk.j1; ++j) {
    const int b = (j - tk.j0) & 1;
    if (j + 1 < tk.j1) {
      issue_keys(j + 1, b ^ 1);
      issue_tile(j + 1, b ^ 1);
    }
    cp_async_commit();
    cp_async_wait<1>();  // digit j's copies are done (this thread's)
    __syncthreads();     // ... and every thread's
    u64 *sm = tiles + b * SM::TILEW;
    const u64 *k0 = keys + b * SM::KEYW;
    const bool ow = own(j);
    if (!ow) {
      tw_ready<TMA>(&twbar, a.tab.err);
      tile_fwd<GT::LOGB, GT::LOGGR, GT::PR, GT::NT, true, RL>(sm, tws, mi.m);
    }
    if (!mbar_wait(&keybar[b], ((j - tk.j0) >> 1) & 1)) atomicExch(a.tab.err, 1);
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      const int e = threadIdx.x + k * NT;
      if (TILE % NT != 0 && e >= TILE) break;
      const u64 x = sm[(e & (GT::N2 - 1)) * GT::PR + (e >> GT::LOGB)];
      u64 y;
      if (ow) {
        y = shoup(x, mi.r1, mi.r1s, mi.m);  // d_t in Montgomery form, [0, 2m)
        if (!lazy) y = csub(y, mi.m);
      } else if (lazy) {
        y = x;
      } else {
        y = fwd_canon(x, mi.m, mi.mu, cls);
      }
      const u64 ka = k0[e], kb = k0[TILE + e];
      if (WIDE) {
        mac128(w0[k], y, ka);
        mac128(w1[k], y, kb);
      } else {
        U128 p0 = {0, 0}, p1 = {0, 0};
        mac128(p0, y, ka);
        mac128(p1, y, kb);
        const u64 a0v = s0[k] + redc(p0, mi.m, mi.minv), a1v = s1[k] + redc(p1, mi.m, mi.minv);
        s0[k] = a0v >= m2 ? a0v - m2 : a0v;
        s1[k] = a1v >= m2 ? a1v - m2 : a1v;
      }
    }
    __syncthreads();  // buffers b are free for digit j + 2
  }
  u64 *a0 = acc + (size_t)t * N + off0;
  u64 *a1 = acc + ((size_t)a.qp + t) * N + off0;
#pragma unroll
  for (int k = 0; k < EPT; ++k) {
    const int e = threadIdx.x + k * NT;
    if (TILE % NT != 0 && e >= TILE) break;
    u64 r0v, r1v;
    if (WIDE) {
      r0v = csub(redc(w0[k], mi.m, mi.minv), mi.m);
      r1v = csub(redc(w1[k], mi.m, mi.minv), mi.m);
    } else {
      r0v = csub(s0[k], mi.m);
      r1v = csub(s1[k], mi.m);
    }
    if (!tk.first) {
      r0v = addmod(r0v, a0[e], mi.m);
      r1v = addmod(r1v, a1[e], mi.m);
    }
    a0[e] = r0v;
    a1[e] = r1v;
  }
}

template <int LOGN, int RL, int PRO>
__global__ void __launch_bounds__(GeoT<LOGN, RL, 1>::NT,
                                  min_blocks(GeoT<LOGN, RL, 1>::NT,
                                             RL == 4 ? 384 : RL == 2 ? 1024 : 768))
    k_fwd_row_keymult(KArgs a, JobSet js, WsOff wo, Tasks tk) {
  extern __shared__ __align__(16) unsigned char raw[];
  // Targets in reverse: the P-limb targets, listed last, have no digit of their own (one
  // more NTT per CTA), so starting them first shortens the tail of multi-wave launches
  // (measured on GB300 at (4, 2^16, 35): 125 -> 121 us for this launch).
  const int by = gridDim.y - 1 - blockIdx.y;
  __shared__ u64 cst[kMaxLimbs];
  keymult_body<LOGN, RL, PRO>(a, js.j[blockIdx.z], wo, tk, blockIdx.x, by, raw, cst);
  pdl_trigger();  // the next kernel may launch once every CTA is here
}

// ModDown row pass fused with the final scaling, both polynomials c = 0, 1 of
// limb i (TASK_DOWN1) in one CTA (shared twiddles):
//   out_c[i] = (acc_c[i] - NTT(BConv_{P->Q}(c))[i]) * P^-1 mod q_i.
template <int LOGN, int RL, int PRO, bool TMA = true>
__device__ __forceinline__ void moddown_body(const KArgs &a, const JobPtr &jp, const WsOff &wo,
                                             const Tasks &tk, int bx, int by,
                                             unsigned char *raw, u64 *cst) {
  using GT = GeoT<LOGN, RL, 1>;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *sm = tile_ptr<GT, false>(raw);
  const u64 *vp = jp.ws + wo.vp, *tmp2 = jp.ws + wo.tmp2, *acc = jp.ws + wo.acc;
  const uint32_t w = decode(a, tk, by);
  const int i = task_limb(w), blk = bx, r0 = blk * GT::GR;
  const u64 m = a.tab.mod[i].m;
  const ulonglong2 pv = a.tab.pinv[i];
  const size_t N = a.N;
  const size_t off0 = (size_t)r0 << GT::LOGB;
  // The NTT output z enters the scaling lazy: below kFwdLazy * m (fast butterflies) or,
  // after one conditional subtraction, below 8m (mid) or 2m (exact); acc + zb - z is then
  // positive and below (kFwdLazy + 1) m, 9m or 3m < 2^64, and the Shoup product by P^-1
  // takes any word.
  const int cls = mod_class(m);
  const bool fast = cls == CLS_FAST;
  const u64 zs = cls == CLS_MID ? 8 * m : 2 * m, zb = fast ? kFwdLazy * m : zs;
  if (threadIdx.x == 0)
    for (int c = 0; c < 2; ++c) prefetch_l2(acc + ((size_t)c * a.qp + i) * N + off0, GT::TILE * 8);
  __shared__ u64 twbar;
  stage_row_slab<GT, TMA>(tws, row_table<GT>(a.tab.twr_f, i, blk), &twbar);
  pdl_wait();
  for (int c = 0; c < 2; ++c) {
    const uint32_t wc = pack_task(i, c, task_slot(w) + c * tk.span);
    if (GT::LOGA == 0)
      produce<GT, PRO, false>(a, sm, cst, wc, vp, tmp2, r0);
    else
      produce<GT, PRO_LOAD, false>(a, sm, cst, wc, vp, tmp2, r0);
    __syncthreads();
    tw_ready<TMA>(&twbar, a.tab.err);
    tile_fwd<GT::LOGB, GT::LOGGR, GT::PR, GT::NT, true, RL>(sm, tws, m);
    const u64 *ac = acc + ((size_t)c * a.qp + i) * N + off0;
    const size_t ob = ((size_t)c * a.nq + i) * N + off0;
    u64 *o = jp.out + ob;
    if ((jp.addmask >> c) & 1) {
      const u64 *ad = jp.add + ob;
#pragma unroll
      for (int k = 0; k < GT::EPT; ++k) {
        const int e = threadIdx.x + k * GT::NT;
        if (GT::TILE % GT::NT != 0 && e >= GT::TILE) break;
        const int g = e >> GT::LOGB, x = e & (GT::N2 - 1);
        const u64 z = fast ? sm[x * GT::PR + g] : csub(sm[x * GT::PR + g], zs);
        o[e] = addmod(csub(shoup(ac[e] + zb - z, pv.x, pv.y, m), m), ad[e], m);
      }
    } else {
#pragma unroll
      for (int k = 0; k < GT::EPT; ++k) {
        const int e = threadIdx.x + k * GT::NT;
        if (GT::TILE % GT::NT != 0 && e >= GT::TILE) break;
        const int g = e >> GT::LOGB, x = e & (GT::N2 - 1);
        const u64 z = fast ? sm[x * GT::PR + g] : csub(sm[x * GT::PR + g], zs);
        o[e] = csub(shoup(ac[e] + zb - z, pv.x, pv.y, m), m);
      }
    }
    __syncthreads();
  }
}

// Shared memory of the pipelined ModDown row pass: the row twiddles, the two
// polynomials' NTT tiles (odd pitch) and their accumulator tiles (contiguous).
template <class GT>
struct MdSmem {
  static constexpr int TW = GT::TWS * 16;
  static constexpr int TILEW = GT::N2 * GT::PR;
  static constexpr int BYTES = TW + 2 * TILEW * 8 + 2 * GT::TILE * 8;
};

// moddown_body for N >= 2^13 (persistent batch) with both polynomials' input tiles (cp.async into the odd
// pitch) and accumulator tiles (TMA bulk copies on a barrier) copied into shared memory
// at the start: the copies of c = 1 and of the accumulators are in flight while c = 0
// is transformed. Same arithmetic and result.
template <int LOGN, int RL>
__device__ __forceinline__ void moddown_pipe_body(const KArgs &a, const JobPtr &jp,
                                                  const WsOff &wo, const Tasks &tk, int bx,
                                                  int by, unsigned char *raw) {
  using GT = GeoT<LOGN, RL, 1>;
  using SM = MdSmem<GT>;
  constexpr bool TMA = true;
  constexpr int EPT = GT::EPT, TILE = GT::TILE, NT = GT::NT;
  ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(raw);
  u64 *tiles = reinterpret_cast<u64 *>(raw + SM::TW);
  u64 *accs = tiles + 2 * SM::TILEW;
  const u64 *tmp2 = jp.ws + wo.tmp2, *acc = jp.ws + wo.acc;
  const uint32_t w = decode(a, tk, by);
  const int i = task_limb(w), blk = bx, r0 = blk * GT::GR;
  const u64 m = a.tab.mod[i].m;
  const ulonglong2 pv = a.tab.pinv[i];
  const size_t N = a.N;
  const size_t off0 = (size_t)r0 << GT::LOGB;
  // the NTT output enters the scaling lazy, as in moddown_body
  const int cls = mod_class(m);
  const bool fast = cls == CLS_FAST;
  const u64 zs = cls == CLS_MID ? 8 * m : 2 * m, zb = fast ? kFwdLazy * m : zs;
  __shared__ u64 twbar;
  stage_row_slab<GT, TMA>(tws, row_table<GT>(a.tab.twr_f, i, blk), &twbar);
  pdl_wait();
  // the accumulator tiles (contiguous): one TMA bulk copy each, on one barrier
  __shared__ u64 accbar;
  if (threadIdx.x == 0) {
    mbar_init(&accbar, 1);
    mbar_expect_tx(&accbar, 2 * TILE * 8);
    for (int c = 0; c < 2; ++c)
      bulk_g2s(accs + c * TILE, acc + ((size_t)c * a.qp + i) * N + off0, TILE * 8, &accbar);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const u64 *src = tmp2 + (size_t)(task_slot(w) + c * tk.span) * N + off0;
    u64 *st = tiles + c * SM::TILEW;
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      const int e = threadIdx.x + k * NT;
      if (TILE % NT != 0 && e >= TILE) break;
      cp_async8(st + (e & (GT::N2 - 1)) * GT::PR + (e >> GT::LOGB), src + e);
    }
    cp_async_commit();
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (c == 0)
      cp_async_wait<1>();
    else
      cp_async_wait<0>();
    __syncthreads();
    u64 *sm = tiles + c * SM::TILEW;
    const u64 *sa = accs + c * TILE;
    tw_ready<TMA>(&twbar, a.tab.err);
    tile_fwd<GT::LOGB, GT::LOGGR, GT::PR, GT::NT, true, RL>(sm, tws, m);
    if (c == 0 && !mbar_wait(&accbar, 0)) atomicExch(a.tab.err, 1);
    const size_t ob = ((size_t)c * a.nq + i) * N + off0;
    u64 *o = jp.out + ob;
    const bool add = (jp.addmask >> c) & 1;
    const u64 *ad = jp.add + ob;
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      const int e = threadIdx.x + k * NT;
      if (TILE % NT != 0 && e >= TILE) break;
      const u64 zr = sm[(e & (GT::N2 - 1)) * GT::PR + (e >> GT::LOGB)];
      const u64 z = fast ? zr : csub(zr, zs);
      u64 r = csub(shoup(sa[e] + zb - z, pv.x, pv.y, m), m);
      if (add) r = addmod(r, ad[e], m);
      o[e] = r;
    }
  }
}

template <int LOGN, int RL, int PRO>
__global__ void __launch_bounds__(GeoT<LOGN, RL, 1>::NT,
                                  min_blocks(GeoT<LOGN, RL, 1>::NT, RL == 4 ? 0 : 1024))
    k_fwd_row_moddown(KArgs a, JobSet js, WsOff wo, Tasks tk) {
  extern __shared__ __align__(16) unsigned char raw[];
  // host-buffer operation: let the next one's input pass (which reads host memory and
  // does not wait for this kernel before it ends) start while this one writes its result
  // to host memory
  if (js.j[blockIdx.z].dsrc) pdl_trigger();
  __shared__ u64 cst[kMaxLimbs];
  moddown_body<LOGN, RL, PRO>(a, js.j[blockIdx.z], wo, tk, blockIdx.x, blockIdx.y, raw, cst);
  pdl_trigger();  // the next kernel may launch once every CTA is here
}

// ---------------------------------------------------------------------------
// Launchers for one N and radix.

cudaError_t smem_opt_in(const void *kernel, int bytes);

template <class K>
inline cudaError_t smem_attr(K kernel, int bytes) {
  return smem_opt_in(reinterpret_cast<const void *>(kernel), bytes);
}

inline KArgs args_of(const ks_context *c) { return make_args(c); }

// Whether a launch of `threads` threads lets its dependent launch as soon as its own CTAs
// have all started (see pdl_trigger): when it is more than a wave at the kernels' 768
// threads per SM. (Half of that: (4, 2^16, 35) in four chunks 672 -> 716 us, whose launches
// are about a wave; twice: (4, 2^16, 35) 344 -> 349 us.)
inline int early_rule(size_t threads) { return threads > (size_t)kSms * 768 ? 1 : 0; }

// launch_pdl of a kernel whose first argument is its KArgs, with the early rule applied.
template <class... KT, class... AT>
inline cudaError_t launch_rule(void (*kernel)(KArgs, KT...), dim3 grid, dim3 block, size_t smem,
                               cudaStream_t s, const ks_context *c, AT &&...args) {
  KArgs a = args_of(c);
  a.early = early_rule((size_t)grid.x * grid.y * grid.z * block.x);
  return launch_pdl(kernel, grid, block, smem, s, a, static_cast<AT &&>(args)...);
}

}  // namespace kern
}  // namespace ks
