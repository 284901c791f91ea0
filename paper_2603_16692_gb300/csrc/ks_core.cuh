// Register-tile NTT core of the two-pass sizes (N >= 2^12, device side).
//
// A thread holds E = 2^RL points of one sub-transform (a row or a column) of M = 2^LOGM
// points; T = M / E threads share it. The LOGM stages run as RL stages in registers, one
// exchange through shared memory, R2 = min(RL, LOGM - RL) more stages in registers, and,
// when S = LOGM - RL - R2 stages are left, S steps that swap a register-index bit with a
// lane bit by shuffles and run one stage each. Points move to and from global memory
// straight from registers on the side where the thread's points are T apart (forward
// input, inverse output). A row's T <= 32 threads sit in one warp, so a row pass
// synchronises warps only.
//
// Why: the tile-in-shared-memory rounds (ks_ntt.cuh) move every point through shared
// memory once per two (radix 4) or three (radix 8) stages, with a block barrier each
// time: at radix 4 a row pass of 256 points costs 28 shared-memory wavefronts per
// warp-round against 128 cycles of the integer pipe it has to feed, and four block
// barriers. Here one exchange and one barrier-free hand-off serve eight stages.
#pragma once
#include "ks_arith.cuh"
#include "ks_internal.h"
#include "ks_ntt.cuh"

namespace ks {
namespace core {

// log2 of the points per thread of the row pass (rows of 64 points at N = 2^12, 128 at 2^13
// and 2^14, 256 at 2^15 and 2^16, 512 at 2^17). 16 points halve the exchange traffic and the
// instructions around it, but half the threads with 80 registers instead of 64 wait longer
// on memory: at N = 2^16 8 points took (4, 2^16, 35) in four chunks from 674 to 604 us and
// (4, 2^16, 13 limbs up) from 167 to 160, (4, 2^16, 35) 346 -> 348; rows of 512 points do
// not fit a warp at 8.
__host__ __device__ constexpr int row_rl(int logn) { return logn >= 17 ? 4 : 3; }
// ... and of the column pass (columns of 64, 128, 128, 256, 256 points).
__host__ __device__ constexpr int col_rl(int logn) { return geo_loga(logn) == 8 ? 4 : 3; }

template <int LOGM_, int RL_>
struct Sub {
  static constexpr int LOGM = LOGM_, RL = RL_;
  static constexpr int M = 1 << LOGM, E = 1 << RL, T = 1 << (LOGM - RL), LOGT = LOGM - RL;
  static constexpr int R2 = LOGM - RL < RL ? LOGM - RL : RL;
  static constexpr int S = LOGM - RL - R2;
  static constexpr int EX = RL - R2;  // log2 of a thread's groups in the second round
  static constexpr bool LOOP = RL == kRowHead && R2 == RL;  // both rounds as one loop
  static_assert(R2 >= 1 && (S == 0 || EX == 0) && S <= 2, "two register rounds and swaps");
};

// Position of point x of a row in its shared-memory row: 16 points, then two words of
// padding, so that 16-byte accesses at 16-point strides and 8-byte accesses to
// consecutive points are both free of bank conflicts.
__host__ __device__ constexpr int row_pos(int x) { return x + 2 * (x >> 4); }
// Words of a row; rows of T = 8 threads alternate between the bank halves.
template <class SB>
__host__ __device__ constexpr int row_pitch() {
  return SB::M / 16 * 18 + (SB::T == 8 ? 8 : 0);
}

// R stages from local stage LS0 on the register groups (ex, u) = v[ex 2^R + u];
// tw(q, ex, sub): twiddle of stage LS0 + q, block (hi(ex) << q) + sub.
template <int LOGM, int LS0, int R, int EX, int CLS, class TW>
__device__ __forceinline__ void round_fwd(u64 *v, u64 m, TW tw) {
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int half = 1 << (R - 1 - q);
#pragma unroll
    for (int ex = 0; ex < (1 << EX); ++ex)
#pragma unroll
      for (int u = 0; u < (1 << R); ++u) {
        if (u & half) continue;
        const ulonglong2 w = tw(q, ex, u >> (R - q));
        bfly_fwd_c<CLS>(v[(ex << R) + u], v[(ex << R) + u + half], w, m, LS0 + q);
      }
  }
}
// The inverse; mb 2^(LOGM - ls) is the fast class's bias of stage ls (mb = m, or m shifted by
// the stages after ls = LOGM - 1 of a round that runs as stages 0.. of a shorter transform).
template <int LOGM, int LS0, int R, int EX, int CLS, bool NEG, class TW>
__device__ __forceinline__ void round_inv(u64 *v, u64 m, TW tw, u64 mb) {
#pragma unroll
  for (int q = R - 1; q >= 0; --q) {
    const int half = 1 << (R - 1 - q);
#pragma unroll
    for (int ex = 0; ex < (1 << EX); ++ex)
#pragma unroll
      for (int u = 0; u < (1 << R); ++u) {
        if (u & half) continue;
        const ulonglong2 w = tw(q, ex, u >> (R - q));
        bfly_inv_c<CLS, NEG>(v[(ex << R) + u], v[(ex << R) + u + half], w, m,
                             mb << (LOGM - (LS0 + q)));
      }
  }
}

// Exchange register-index bit rb with lane bit lb: afterwards v[r] of a lane whose bit lb
// is l, r's bit rb being b, is the old v[r with bit rb = l] of the lane whose bit lb is b.
template <int RL>
__device__ __forceinline__ void swap_bits(u64 *v, int rb, int lb) {
  const bool up = (threadIdx.x >> lb) & 1;
#pragma unroll
  for (int r = 0; r < (1 << RL); ++r) {
    if ((r >> rb) & 1) continue;
    const int r1 = r | (1 << rb);
    const u64 got = __shfl_xor_sync(0xffffffffu, up ? v[r] : v[r1], 1 << lb);
    if (up)
      v[r] = got;
    else
      v[r1] = got;
  }
}

// After the swaps, register r of thread t holds point t E + low_of(r).
template <class SB>
__host__ __device__ constexpr int low_of(int r) {
  int x = 0;
  for (int j = 0; j < SB::S; ++j) x |= ((r >> (SB::RL - 1 - j)) & 1) << (SB::S - 1 - j);
  for (int k = 0; k < SB::RL - SB::S; ++k) x |= ((r >> k) & 1) << (SB::S + k);
  return x;
}
// The register that holds low point x.
template <class SB>
__host__ __device__ constexpr int reg_of(int x) {
  for (int r = 0; r < SB::E; ++r)
    if (low_of<SB>(r) == x) return r;
  return 0;
}
// Block index of the stage after swap i for (thread t, register r, its bit RL-1-i clear).
template <class SB>
__device__ __forceinline__ int swap_block(int i, int t, int r) {
  int c = (t >> SB::S) << (SB::RL + i);
#pragma unroll
  for (int j = 0; j <= i; ++j) c |= ((t >> (SB::S - 1 - j)) & 1) << (SB::RL - 1 - j + i);
#pragma unroll
  for (int k = 0; k < SB::RL - 1 - i; ++k) c |= ((r >> k) & 1) << (k + i);
#pragma unroll
  for (int j = 0; j < i; ++j) c |= ((r >> (SB::RL - 1 - j)) & 1) << (i - 1 - j);
  return c;
}

// A thread's block index in the second round, group ex.
template <class SB>
__device__ __forceinline__ int hi_of(int t, int ex) {
  return SB::S == 0 ? (t << SB::EX) + ex : t >> SB::S;
}
// Entry of (stage RL + q, block (hi << q) + sub) in a row's slab: row_tw with the parts
// that are known at compile time folded (RL <= 4, so only hi is not).
template <int RL>
__device__ __forceinline__ int row_tw2(int q, int hi, int sub) {
  const int ls = RL + q;
  if (ls < kRowHead) return (1 << ls) - 1 + (hi << q) + sub;
  const int d = ls - kRowHead;
  return (1 << kRowHead) - 1 + (((1 << d) - 1 + (sub & ((1 << d) - 1))) << kRowHead) +
         (hi << (q - d)) + (sub >> d);
}

// Rows and columns whose two register rounds have the same shape (RL = R2 = 4) run them as
// a loop of two over one copy of the code: unrolled, the 64 butterflies of a 256-point
// transform are 20 KB of instructions, more than a scheduler's instruction cache, and the
// warps waited on instruction fetches (no_instruction 2.9 of 11 stalled warps per issue in
// the input iNTT rows at N = 2^16, which ran 27.8 us that way).

// Forward row transform. In: v[u] = point u T + t. Out: v[r] = point t E + low_of(r).
// s: the row's shared-memory row (used for the exchange), tw: the row's slab.
template <class SB, int CLS>
__device__ __forceinline__ void row_fwd(u64 *v, u64 *s, const ulonglong2 *tw, u64 m, int t) {
  constexpr int RL = SB::RL, R2 = SB::R2, S = SB::S, E = SB::E;
  auto exchange = [&] {
    __syncwarp();  // the row's earlier reads are done
#pragma unroll
    for (int u = 0; u < E; ++u) s[row_pos((u << SB::LOGT) + t)] = v[u];
    __syncwarp();
    if constexpr (S == 0) {
      const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(s + row_pos(t * E));
#pragma unroll
      for (int r = 0; r < E; r += 2) {
        const ulonglong2 x = p[r / 2];
        v[r] = x.x;
        v[r + 1] = x.y;
      }
    } else {
      const int base = ((t >> S) << (RL + S)) + (t & ((1 << S) - 1));
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = s[row_pos(base + (r << S))];
    }
  };
  if constexpr (SB::LOOP) {
    // entry e of a round's tree: the head's e, then row_tw2's 15 + 16 e + hi
    const ulonglong2 *w = tw;
    int sh = 0;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      round_fwd<SB::LOGM, 0, RL, 0, CLS>(
          v, m, [&](int q, int, int sub) { return w[((1 << q) - 1 + sub) << sh]; });
      if (k == 0) {
        exchange();
        w = tw + (1 << kRowHead) - 1 + hi_of<SB>(t, 0);
        sh = kRowHead;
      }
    }
  } else {
    round_fwd<SB::LOGM, 0, RL, 0, CLS>(
        v, m, [&](int q, int, int sub) { return tw[(1 << q) - 1 + sub]; });
    exchange();
    round_fwd<SB::LOGM, RL, R2, SB::EX, CLS>(v, m, [&](int q, int ex, int sub) {
      return tw[row_tw2<RL>(q, hi_of<SB>(t, ex), sub)];
    });
  }
#pragma unroll
  for (int i = 0; i < S; ++i) {
    const int rb = RL - 1 - i, ls = RL + R2 + i;
    swap_bits<RL>(v, rb, S - 1 - i);
#pragma unroll
    for (int r = 0; r < E; ++r) {
      if ((r >> rb) & 1) continue;
      bfly_fwd_c<CLS>(v[r], v[r | (1 << rb)], tw[row_tw(ls, swap_block<SB>(i, t, r))], m, ls);
    }
  }
}

// Inverse row transform (mirrored slab: the row's stage-ls block c is entry 2^ls - 1 - c of
// the mirrored row, negated). In: v[r] = point t E + low_of(r). Out: v[u] = point u T + t.
template <class SB, int CLS>
__device__ __forceinline__ void row_inv(u64 *v, u64 *s, const ulonglong2 *tw, u64 m, int t) {
  constexpr int RL = SB::RL, R2 = SB::R2, S = SB::S, E = SB::E;
#pragma unroll
  for (int i = S - 1; i >= 0; --i) {
    const int rb = RL - 1 - i, ls = RL + R2 + i;
#pragma unroll
    for (int r = 0; r < E; ++r) {
      if ((r >> rb) & 1) continue;
      const int c = (1 << ls) - 1 - swap_block<SB>(i, t, r);
      bfly_inv_c<CLS, true>(v[r], v[r | (1 << rb)], tw[row_tw(ls, c)], m,
                            m << (SB::LOGM - ls));
    }
    swap_bits<RL>(v, rb, S - 1 - i);
  }
  auto exchange = [&] {
    __syncwarp();  // the row's earlier reads (the caller's tile) are done
    if constexpr (S == 0) {
      ulonglong2 *p = reinterpret_cast<ulonglong2 *>(s + row_pos(t * E));
#pragma unroll
      for (int r = 0; r < E; r += 2) p[r / 2] = make_ulonglong2(v[r], v[r + 1]);
    } else {
      const int base = ((t >> S) << (RL + S)) + (t & ((1 << S) - 1));
#pragma unroll
      for (int r = 0; r < E; ++r) s[row_pos(base + (r << S))] = v[r];
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < E; ++u) v[u] = s[row_pos((u << SB::LOGT) + t)];
  };
  if constexpr (SB::LOOP) {
    // second round first: entry e of the mirrored tree, bias m 2^(S + 1 ..)
    const ulonglong2 *w = tw + (1 << kRowHead) - 1 + (1 << RL) - 1 - hi_of<SB>(t, 0);
    int sh = kRowHead;
    u64 mb = m << S;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      round_inv<RL, 0, RL, 0, CLS, true>(
          v, m, [&](int q, int, int sub) { return w[((2 << q) - 2 - sub) << sh]; }, mb);
      if (k == 0) {
        exchange();
        w = tw;
        sh = 0;
        mb = m << (S + RL);
      }
    }
  } else {
    round_inv<SB::LOGM, RL, R2, SB::EX, CLS, true>(
        v, m,
        [&](int q, int ex, int sub) {
          return tw[row_tw2<RL>(q, (1 << RL) - 1 - hi_of<SB>(t, ex), (1 << q) - 1 - sub)];
        },
        m);
    exchange();
    round_inv<SB::LOGM, 0, RL, 0, CLS, true>(
        v, m, [&](int q, int, int sub) { return tw[(2 << q) - 2 - sub]; }, m);
  }
}

// The thread's E contiguous points to / from its row in shared memory (16-byte accesses).
template <class SB>
__device__ __forceinline__ void put_row(u64 *s, const u64 *v, int t) {
  ulonglong2 *p = reinterpret_cast<ulonglong2 *>(s + row_pos(t * SB::E));
#pragma unroll
  for (int x = 0; x < SB::E; x += 2)
    p[x / 2] = make_ulonglong2(v[reg_of<SB>(x)], v[reg_of<SB>(x + 1)]);
}
template <class SB>
__device__ __forceinline__ void get_row(u64 *v, const u64 *s, int t) {
  const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(s + row_pos(t * SB::E));
#pragma unroll
  for (int x = 0; x < SB::E; x += 2) {
    const ulonglong2 y = p[x / 2];
    v[reg_of<SB>(x)] = y.x;
    v[reg_of<SB>(x + 1)] = y.y;
  }
}

// Column transforms run in ceil(LOGM / RL) register rounds with an exchange through shared
// memory before each but the first. Round K covers the stages from RL K on: point
// (hi: RL K bits, u: the round's stages, lo: the rest); a thread holds every u of its
// (hi, lo), in the last round of its 2^EX consecutive hi.
template <int LOGM, int RL, int K>
struct ColRound {
  static constexpr int LS0 = RL * K, R = LOGM - LS0 < RL ? LOGM - LS0 : RL, EX = RL - R;
  static constexpr int SUB = LOGM - LS0 - R;
  static constexpr bool LAST = SUB == 0;
  static __device__ __forceinline__ int hi(int t, int ex) {
    return LAST ? (t << EX) + ex : t >> SUB;
  }
  // point of register r = (ex, u)
  static __device__ __forceinline__ int point(int t, int r) {
    const int ex = r >> R, u = r & ((1 << R) - 1);
    return (hi(t, ex) << (R + SUB)) + (u << SUB) + (LAST ? 0 : t & ((1 << SUB) - 1));
  }
};
// Row position of a point in the exchange tile: a pad row after every 2^RL rows, so that
// the last round's threads (2^RL rows apart) start in different banks.
template <int RL>
__device__ __forceinline__ int col_pos(int y) {
  return y + (y >> RL);
}
template <int LOGM, int RL>
__host__ __device__ constexpr int col_rounds() {
  return (LOGM + RL - 1) / RL;
}

// Inverse column transform of column g of a tile of GC columns (tw: the column table, entry
// 2^ls + c). In: v[r] = point ColRound<last>::point(t, r), below 4m (fast; so the biases are
// four times a canonical start's, and the outputs below 2^(LOGM + 3) m), 8m (mid) or 2m
// (exact). Out: v[u] = point u T + t.
// sync(): barrier of the tile's threads.
template <int LOGM, int RL, int GC, int CLS, int K, class SYNC>
__device__ __forceinline__ void col_inv(u64 *v, u64 *s, const ulonglong2 *tw, u64 m, int t, int g,
                                        SYNC sync) {
  using C = ColRound<LOGM, RL, K>;
  auto exchange = [&] {  // from round K's points to round K - 1's
    using P = ColRound<LOGM, RL, K == 0 ? 0 : K - 1>;
#pragma unroll
    for (int r = 0; r < (1 << RL); ++r) s[col_pos<RL>(C::point(t, r)) * GC + g] = v[r];
    sync();
#pragma unroll
    for (int r = 0; r < (1 << RL); ++r) v[r] = s[col_pos<RL>(P::point(t, r)) * GC + g];
  };
  if constexpr (LOGM == 2 * RL) {  // both rounds as one loop (see row_fwd)
    int h = (1 << RL) + C::hi(t, 0);  // entry of (stage q of the round, sub): (h << q) + sub
    u64 mb = 4 * m;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      round_inv<RL, 0, RL, 0, CLS, false>(
          v, m, [&](int q, int, int sub) { return tw[(h << q) + sub]; }, mb);
      if (k == 0) {
        exchange();
        h = 1;
        mb = m << (RL + 2);
      }
    }
  } else {
    round_inv<LOGM, C::LS0, C::R, C::EX, CLS, false>(
        v, m,
        [&](int q, int ex, int sub) {
          return tw[(1 << (C::LS0 + q)) + (C::hi(t, ex) << q) + sub];
        },
        4 * m);
    if constexpr (K > 0) {
      exchange();  // (the next one writes where this thread just read)
      col_inv<LOGM, RL, GC, CLS, K - 1>(v, s, tw, m, t, g, sync);
    }
  }
}
// Forward column transform. In: v[u] = point u T + t (below 2m). Out: v[r] = point
// ColRound<last>::point(t, r), lazy. The caller syncs before the tile is used again.
template <int LOGM, int RL, int GC, int CLS, int K, class SYNC>
__device__ __forceinline__ void col_fwd(u64 *v, u64 *s, const ulonglong2 *tw, u64 m, int t, int g,
                                        SYNC sync) {
  using C = ColRound<LOGM, RL, K>;
  round_fwd<LOGM, C::LS0, C::R, C::EX, CLS>(v, m, [&](int q, int ex, int sub) {
    return tw[(1 << (C::LS0 + q)) + (C::hi(t, ex) << q) + sub];
  });
  if constexpr (!C::LAST) {
    using P = ColRound<LOGM, RL, K + 1>;
#pragma unroll
    for (int r = 0; r < (1 << RL); ++r) s[col_pos<RL>(C::point(t, r)) * GC + g] = v[r];
    sync();
#pragma unroll
    for (int r = 0; r < (1 << RL); ++r) v[r] = s[col_pos<RL>(P::point(t, r)) * GC + g];
    col_fwd<LOGM, RL, GC, CLS, K + 1>(v, s, tw, m, t, g, sync);
  }
}

// Words of a column tile's exchange buffer.
template <int LOGM, int GC, int RL>
__host__ __device__ constexpr int col_words() {
  return ((1 << LOGM) + ((1 << LOGM) >> RL)) * GC;
}

}  // namespace core
}  // namespace ks
