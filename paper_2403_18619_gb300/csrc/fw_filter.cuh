// Filtered min-plus for element types whose relaxation is expensive (fp64: the
// narrow FP64 pipe): a 16-bit pass finds the entries that can improve, and only
// those are relaxed exactly.
//
// Operand tiles are also kept as 13-bit lower bounds, q = floor(v * 2^e) with
// one exponent e per round (the closed pivot's largest finite entry chooses
// it), in the layout of the 16-bit keys (h_unit).  core_h then gives
//     F = min over kk of q(A[row][kk]) + q(B[kk][col])
// at two relaxations per instruction.  F * 2^-e bounds every exact sum from
// below, also after rounding (the bound is representable and rounding is
// monotone), so an entry with F * 2^-e >= its value cannot improve.  For the
// others, every step whose bound is at most F + 2 is summed exactly, in the
// element type: the true sum of F's step lies below F + 2, so no other step
// can be smaller or, equal, be rounded to the same value.  Ties go to the
// first step, as in a relaxation in order: distances and predecessors are
// those of the exact kernel, bit for bit.
//   * a finite value above the range is 8191, which still bounds it from below
//     (but not from above: with F >= 8191 every finite step is summed);
//   * INF is 16383: a sum with it is at least that;
//   * negative entries are flagged per tile, which is then relaxed over every step
//     of every entry (relax_exact);
//   * so is a warp's part of a tile whose candidates have so many steps to sum that
//     this is quicker: where the bounds say little, because the entries of a tile are
//     far larger or smaller than those that chose the exponent (a vertex far from all
//     others, a large finite weight for a missing edge).  The tiles of a round that a
//     warp takes after such a one are not filtered at all, but for one in four
//     (skip_filter).
#pragma once

#include "fw_device.cuh"
#include "fw_quad.cuh"

namespace fwk {

// One tile to relax: its operands exactly and as bounds, and where it goes.
template <typename T>
struct FilterTask {
  const T* A;            // exact operands, [row][kk] and [kk][col] (BS x BS, any memory)
  const T* B;
  const T* old;          // the tile's values before, BS x BS in shared memory
  const uint32_t* Ah;    // their 16-bit bounds in shared memory
  const uint32_t* Bh;
  const int32_t* Psrc;   // predecessors of B's rows, [kk][col]
  T* D;                  // the tile in the matrix
  int32_t* P;            // null: distance-only
  int64_t ld;
  int nrow, ncol, kn;    // valid rows, columns and steps
  bool diag;             // the tile lies on the diagonal
  bool neg;              // an operand has a negative entry
  QScale q;
  int* status;
};

// Threshold of a candidate's steps: F + 2; every finite step where F does not
// bound its step's sum from above.
__device__ __forceinline__ unsigned step_threshold(unsigned F) {
  return F >= kQMax ? kQInf - 1 : F + 2;
}

// The operand units that hold a step at or below the threshold: bit w4 for the
// low halves of unit w4, bit 16 + w4 for the high ones (bit 15 of a half is
// free in the sums, so that subtracting one from thr + 2^15 borrows from
// nothing above).
template <int BS>
__device__ __forceinline__ uint32_t scan_units(const uint32_t* pa, const uint32_t* pb,
                                               unsigned thr) {
  const uint32_t thr2 = thr * 0x10001u | 0x80008000u;
  uint32_t flags = 0;
#pragma unroll 4
  for (int w4 = 0; w4 < BS / 8; ++w4) {
    const uint4 a = *reinterpret_cast<const uint4*>(pa + w4 * Geo<BS>::TM * 64);
    const uint4 b = *reinterpret_cast<const uint4*>(pb + w4 * Geo<BS>::TM * 64);
    const uint32_t m = __vminu2(__vimin3_u16x2(a.x + b.x, a.y + b.y, a.z + b.z), a.w + b.w);
    flags |= (thr2 - m) >> (15 - w4) & 0x10001u << w4;
  }
  return flags;
}

// Calls hit(kk) for the steps of the lowest flagged unit half at or below the
// threshold, and clears its flag.
template <int BS, class F>
__device__ __forceinline__ void next_hits(uint32_t& flags, const uint32_t* pa, const uint32_t* pb,
                                          unsigned thr, F&& hit) {
  const int bit = __ffs((int)flags) - 1, w4 = bit & 15, half = bit >> 4;
  flags &= flags - 1;
  const uint4 a = *reinterpret_cast<const uint4*>(pa + w4 * Geo<BS>::TM * 64);
  const uint4 b = *reinterpret_cast<const uint4*>(pb + w4 * Geo<BS>::TM * 64);
  const uint32_t s[4] = {a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if ((s[e] >> (16 * half) & 0xffffu) <= thr) hit(kk_of<BS>(w4 * 4 + e, half));
}

// Element of an exact operand: kGmem: in global memory, written by other CTAs.
template <bool kGmem, typename T>
__device__ __forceinline__ T operand(const T* p) {
  if constexpr (kGmem) return __ldcg(p);
  else return *p;
}

// Two neighbouring elements (8 bytes each, 16-byte aligned).
template <bool kGmem, typename T>
__device__ __forceinline__ void load_pair(T* dst, const T* src) {
  static_assert(sizeof(T) == 8, "16 bytes");
  int4 v;
  if constexpr (kGmem) v = __ldcg(reinterpret_cast<const int4*>(src));
  else v = *reinterpret_cast<const int4*>(src);
  const long long w[2] = {(long long)(((unsigned long long)(unsigned)v.y << 32) | (unsigned)v.x),
                          (long long)(((unsigned long long)(unsigned)v.w << 32) | (unsigned)v.z)};
#pragma unroll
  for (int e = 0; e < 2; ++e) dst[e] = *reinterpret_cast<const T*>(&w[e]);
}

template <typename T>
__device__ __forceinline__ void store_relaxed(const FilterTask<T>& f, int row, int col, T v,
                                              int32_t pred) {
  f.D[row * f.ld + col] = v;
  if (f.P) f.P[row * f.ld + col] = pred;
  if (f.diag && row == col && v < T(0)) atomicOr(f.status, kStNegCycle);
}

// The few candidates with three or more steps to sum, one per lane: item as
// in refine_list (on: this lane has one).
template <typename T, int BS, bool kGmem>
__device__ __noinline__ void refine_many(const FilterTask<T>& f, uint32_t item, bool on) {
  if (!on) return;
  const int row = item & 127u, col = item >> 7 & 127u;
  const unsigned thr = step_threshold(item >> 14);
  const uint32_t* const pa = f.Ah + unit_of<BS>(row);
  const uint32_t* const pb = f.Bh + unit_of<BS>(col);
  uint32_t flags = scan_units<BS>(pa, pb, thr);
  T best = f.old[row * BS + col];
  int arg = -1;
  // a unit half (four steps) at a time, its operands loaded together
  while (flags) {
    int kk[4] = {0, 0, 0, 0};  // n of them
    int n = 0;
    next_hits<BS>(flags, pa, pb, thr, [&](int k) {
      kk[0] = n == 0 ? k : kk[0];
      kk[1] = n == 1 ? k : kk[1];
      kk[2] = n == 2 ? k : kk[2];
      kk[3] = n == 3 ? k : kk[3];
      ++n;
    });
    T s[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      s[e] = e < n && kk[e] < f.kn
                 ? operand<kGmem>(f.A + row * BS + kk[e]) + operand<kGmem>(f.B + kk[e] * BS + col)
                 : Num<T>::inf();
    // (the first step of the smallest sum, whatever the order of the visits)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (relax_lt<T>(s[e], best) || (e < n && arg >= 0 && s[e] == best && kk[e] < arg)) {
        best = s[e];
        arg = kk[e];
      }
  }
  if (arg >= 0)
    store_relaxed(f, row, col, best, f.P ? __ldcg(f.Psrc + arg * BS + col) : 0);
}

// Unit halves (four steps) of a warp's many-step candidates from which on all of its
// 512 entries are relaxed over all 16 units' halves each, 8192 of them.  Halves that
// are gathered cost about eight times one that is streamed: 700, 1024, 1600 and
// 2048 halves gave n = 700 on a grid 2.49, 2.54, 3.19 and 3.6 ms, a grid of n = 4096
// 18.9, 18.9, 24.7 and 28.5, n = 4096 uniform 26.3, 26.3, 26.9 and 27.4, n = 3000
// uniform without predecessors 11.8, 11.7, 11.7 and 12.0.
constexpr int kMaxWork = 1024;

// Exact relaxation of the `total` candidates of one warp (list: row | col << 7
// | F << 14).  First, every lane scans the bounds of its candidate's row and
// column for the steps to sum and puts them in place of F; then four
// candidates per lane are summed at a time, so that the loads of their
// operands (global memory, for a remaining tile) overlap.  Most candidates
// have one step; those with more than two are set aside and taken together.
// False, with nothing stored, if these have more than kMaxWork halves to sum.
template <typename T, int BS, bool kGmem>
__device__ __noinline__ bool refine_list(const FilterTask<T>& f, uint32_t* list, int total) {
  const int lane = threadIdx.x & 31;
  const uint32_t* const Ah = f.Ah;
  const uint32_t* const Bh = f.Bh;
  const int kn = f.kn;
  uint32_t aside = 0;   // lane's candidate set aside
  int naside = 0;       // lanes that hold one
  int work = 0;         // unit halves (four steps) of the candidates set aside
#pragma unroll 1
  for (int i0 = 0; i0 < total; i0 += 32) {
    const int i = i0 + lane;
    uint32_t item = 0, all = 0;
    bool many = false;
    if (i < total) {
      item = list[i];
      const unsigned thr = step_threshold(item >> 14);
      const uint32_t* const pa = Ah + unit_of<BS>((int)(item & 127u));
      const uint32_t* const pb = Bh + unit_of<BS>((int)(item >> 7 & 127u));
      uint32_t flags = all = scan_units<BS>(pa, pb, thr);
      int n = 0, k1 = 0, k2 = 0;
      while (flags && n < 3)
        next_hits<BS>(flags, pa, pb, thr, [&](int kk) {
          if (kk >= kn) return;
          k2 = n == 1 ? kk : k2;
          k1 = n == 0 ? kk : k1;
          ++n;
        });
      many = n > 2;
      list[i] = (item & 0x3fffu) | (uint32_t)k1 << 14 | (uint32_t)k2 << 21 |
                (uint32_t)(many ? 0 : n) << 28;
      if (many) list[i] = item | 1u << 31;
    }
    if (__any_sync(0xffffffffu, many)) {
      work += __reduce_add_sync(0xffffffffu, many ? __popc(all) : 0);
      if (work > kMaxWork) return false;
    }
  }
#pragma unroll 1
  for (int i0 = 0; work && i0 < total; i0 += 32) {
    const uint32_t item = i0 + lane < total ? list[i0 + lane] : 0u;
    for (unsigned m = __ballot_sync(0xffffffffu, item >> 31); m; m &= m - 1) {
      const uint32_t got = __shfl_sync(0xffffffffu, item, __ffs((int)m) - 1);
      if (lane == naside) aside = got & 0x7fffffffu;
      if (++naside == 32) {
        refine_many<T, BS, kGmem>(f, aside, true);
        naside = 0;
      }
    }
  }
  if (naside) refine_many<T, BS, kGmem>(f, aside, lane < naside);
  const T* const A = f.A;
  const T* const B = f.B;
  const int32_t* const Psrc = f.P ? f.Psrc : nullptr;
#pragma unroll 1
  for (int i0 = lane; i0 < total; i0 += 128) {
    constexpr int I = 4;
    uint32_t item[I];
    T s1[I], s2[I], best[I];
    int arg[I];
    int32_t pred[I];
#pragma unroll
    for (int u = 0; u < I; ++u) item[u] = i0 + 32 * u < total ? list[i0 + 32 * u] : 0u;
#pragma unroll
    for (int u = 0; u < I; ++u) {
      const int row = item[u] & 127u, col = item[u] >> 7 & 127u;
      const int k1 = item[u] >> 14 & 127u, k2 = item[u] >> 21 & 127u, n = item[u] >> 28 & 3u;
      const bool one = !(item[u] >> 31);  // (not one set aside)
      s1[u] = s2[u] = Num<T>::inf();
      best[u] = f.old[row * BS + col];
      if (n >= 1 && one) s1[u] = operand<kGmem>(A + row * BS + k1) + operand<kGmem>(B + k1 * BS + col);
      if (n >= 2 && one) s2[u] = operand<kGmem>(A + row * BS + k2) + operand<kGmem>(B + k2 * BS + col);
    }
#pragma unroll
    for (int u = 0; u < I; ++u) {
      const int col = item[u] >> 7 & 127u;
      const int k1 = item[u] >> 14 & 127u, k2 = item[u] >> 21 & 127u;
      arg[u] = -1;
      pred[u] = 0;
      // (steps that are not there sum to INF)
      if (relax_lt<T>(s1[u], best[u])) { best[u] = s1[u]; arg[u] = k1; }
      if (relax_lt<T>(s2[u], best[u]) || (arg[u] >= 0 && s2[u] == best[u] && k2 < arg[u])) {
        best[u] = s2[u];
        arg[u] = k2;
      }
      if (Psrc && arg[u] >= 0) pred[u] = __ldcg(Psrc + arg[u] * BS + col);
    }
#pragma unroll
    for (int u = 0; u < I; ++u)
      if (arg[u] >= 0)
        store_relaxed(f, item[u] & 127u, item[u] >> 7 & 127u, best[u], pred[u]);
  }
  return true;
}

// Candidates of a warp from the minima of core_h (two halves per entry), as the
// list of refine_list: one word per entry of the warp's part of the tile.
// Returns their number.  Whole warps.
template <typename T, int BS>
__device__ __forceinline__ int find_candidates(const FilterTask<T>& f,
                                               const uint32_t (&acc)[Geo<BS>::TM][Geo<BS>::TM],
                                               int tx, int ty, uint32_t* list) {
  using Gm = Geo<BS>;
  constexpr int TM = Gm::TM, G = Gm::G;
  const int lane = threadIdx.x & 31;
  const QScale q = f.q;
  const int nrow = f.nrow, ncol = f.ncol;
  // the list entry by entry, all lanes' of one before the next: neighbours in
  // it share rows (their bounds are then read by broadcast) and lie in few row
  // segments
  const uint32_t at = (uint32_t)(ty * G) | (uint32_t)(tx * G) << 7;
  const unsigned below = (1u << lane) - 1u;
  int total = 0;
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lr = Gm::idx(ty, m), lc = g * Gm::SPAN + tx * G;
      T v[G];
      vload_s<G>(v, f.old + lr * BS + lc);
#pragma unroll
      for (int e = 0; e < G; ++e) {
        const uint32_t mm = h_min2(acc[m][g * G + (e & ~1)], acc[m][g * G + (e | 1)]);
        const unsigned F = e & 1 ? mm >> 16 : mm & 0xffffu;
        const bool on = F < kQInf && Quant<T>::may_improve(F, v[e], q) && lr < nrow && lc + e < ncol;
        const unsigned all = __ballot_sync(0xffffffffu, on);
        if (on)
          list[total + __popc(all & below)] =
              at + ((uint32_t)Gm::idx(0, m) | (uint32_t)Gm::idx(0, g * G + e) << 7) + (F << 14);
        total += __popc(all);
      }
    }
  return total;
}

// Exact relaxation of a lane's entries over every step in order, with a strict
// compare, on operands read in place (from L2 for a remaining tile: 192 KB a tile,
// far less than the narrow FP64 pipe leaves time for).  Bound by that pipe, as the
// exact kernel: with a vertex at 1e9 in every block of 64 and its edges as likely
// as not, n = 4096 took 405 ms when every entry was refined step by step, 133 with
// the exact kernel, 70.5 now (n = 2048: 52, 17.1, 10.5; n = 1500: 23.1, 7.6, 7.4;
// n = 700: 9.8, 2.87, 2.85).
template <typename T, int BS, bool kGmem>
__device__ __forceinline__ void relax_exact(const FilterTask<T>& f, int tx, int ty) {
  using Gm = Geo<BS>;
  constexpr int TM = Gm::TM, G = Gm::G;
  static_assert(Gm::NG == 1 && sizeof(T) == 8, "one group of 8-byte columns per lane");
  T best[TM][TM];
  int arg[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    vload_s<G>(best[m], f.old + Gm::idx(ty, m) * BS + tx * G);
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) arg[m][nn] = -1;
  }
  const T* const A = f.A + Gm::idx(ty, 0) * BS;
  const T* const B = f.B + tx * G;
  const int kn = f.kn;
  // two steps at a time: an operand row's steps are neighbours in memory
#pragma unroll 1
  for (int k0 = 0; k0 < kn; k0 += 2) {
    T a[TM][2], b[2][G];
#pragma unroll
    for (int m = 0; m < TM; ++m) load_pair<kGmem>(a[m], A + m * BS + k0);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < G; e += 2) load_pair<kGmem>(b[h] + e, B + (k0 + h) * BS + e);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (k0 + h >= kn) break;  // (past the last vertex the operands may hold anything)
#pragma unroll
      for (int m = 0; m < TM; ++m)
#pragma unroll
        for (int nn = 0; nn < TM; ++nn) {
          const T s = a[m][h] + b[h][nn];
          const bool lt = relax_lt<T>(s, best[m][nn]);
          best[m][nn] = lt ? s : best[m][nn];
          arg[m][nn] = lt ? k0 + h : arg[m][nn];
        }
    }
  }
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
    int32_t pred[TM];
#pragma unroll
    for (int nn = 0; nn < TM; ++nn)
      pred[nn] = f.P && arg[m][nn] >= 0 ? __ldcg(f.Psrc + arg[m][nn] * BS + tx * G + nn) : 0;
#pragma unroll
    for (int nn = 0; nn < TM; ++nn)
      if (arg[m][nn] >= 0 && lr < f.nrow && tx * G + nn < f.ncol)
        store_relaxed(f, lr, tx * G + nn, best[m][nn], pred[nn]);
  }
}

// A warp's part of a tile, from the minima of core_h.  False if it is to be relaxed
// over every step instead (relax_exact).
template <typename T, int BS, bool kGmem>
__device__ __forceinline__ bool refine_tile(const FilterTask<T>& f,
                                            const uint32_t (&acc)[Geo<BS>::TM][Geo<BS>::TM], int tx,
                                            int ty, uint32_t* list) {
  if (f.neg) return false;
  const int total = find_candidates<T, BS>(f, acc, tx, ty, list);
  if (total == 0) return true;
  __syncwarp();
  const bool done = refine_list<T, BS, kGmem>(f, list, total);
  __syncwarp();
  return done;
}

// Whether a warp relaxes a tile of round r over every step without asking its
// bounds: it did so in the end with a tile of this round (`exact`: the round of the
// latest such tile).  Every fourth tile asks all the same.  (Asking every tile:
// n = 4096 with far vertices and a coarse exponent 196 ms instead of 136; skipping
// in the round after as well: n = 4096 uniform 27.2 ms instead of 26.9.)
__device__ __forceinline__ bool skip_filter(int exact, int r, int ti, int tj) {
  return r <= exact && ((ti + tj) & 3);
}

}  // namespace fwk
