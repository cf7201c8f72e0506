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
//   * negative entries (only a negative cycle has them) are flagged per tile,
//     and every step of every entry is then summed.
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
  const int32_t* Psrc;   // predecessors of B's rows, [kk][col]; null: via codes
  T* D;                  // the tile in the matrix
  int32_t* P;            // null: distance-only
  int64_t ld;
  int nrow, ncol, kn;    // valid rows, columns and steps
  int r, bs;             // round, block size
  bool diag;             // the tile lies on the diagonal
  bool neg;              // an operand has a negative entry
  QScale q;
  int* status;
};

// Threshold of a candidate's steps: F + 2; every finite step where F does not
// bound its step's sum from above; every step beside a negative entry.
__device__ __forceinline__ unsigned step_threshold(unsigned F, bool neg) {
  return neg ? 0x7fffu : F >= kQMax ? kQInf - 1 : F + 2;
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

template <typename T>
__device__ __forceinline__ void store_relaxed(const FilterTask<T>& f, int row, int col, T v,
                                              int arg, int32_t pred) {
  f.D[row * f.ld + col] = v;
  if (f.P) f.P[row * f.ld + col] = f.Psrc ? pred : via_code((int64_t)f.r * f.bs + arg);
  if (f.diag && row == col && v < T(0)) atomicOr(f.status, kStNegCycle);
}

// The few candidates with three or more steps to sum, one per lane: item as
// in refine_list (on: this lane has one).
template <typename T, int BS, bool kGmem>
__device__ __noinline__ void refine_many(const FilterTask<T>& f, uint32_t item, bool on) {
  if (!on) return;
  const int row = item & 127u, col = item >> 7 & 127u;
  const unsigned thr = step_threshold(item >> 14, f.neg);
  const uint32_t* const pa = f.Ah + unit_of<BS>(row);
  const uint32_t* const pb = f.Bh + unit_of<BS>(col);
  uint32_t flags = scan_units<BS>(pa, pb, thr);
  T best = f.old[row * BS + col];
  int arg = -1;
  // a unit half (four steps) at a time, its operands loaded together
  while (flags) {
    int kk[4];
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
    store_relaxed(f, row, col, best, arg, f.P && f.Psrc ? __ldcg(f.Psrc + arg * BS + col) : 0);
}

// Exact relaxation of the `total` candidates of one warp (list: row | col << 7
// | F << 14).  First, every lane scans the bounds of its candidate's row and
// column for the steps to sum and puts them in place of F; then four
// candidates per lane are summed at a time, so that the loads of their
// operands (global memory, for a remaining tile) overlap.  Most candidates
// have one step; those with more than two are set aside and taken together.
template <typename T, int BS, bool kGmem>
__device__ __noinline__ void refine_list(const FilterTask<T>& f, uint32_t* list, int total) {
  const int lane = threadIdx.x & 31;
  const uint32_t* const Ah = f.Ah;
  const uint32_t* const Bh = f.Bh;
  const int kn = f.kn;
  const bool neg = f.neg;
  uint32_t aside = 0;   // lane's candidate set aside
  int naside = 0;       // lanes that hold one
#pragma unroll 1
  for (int i0 = 0; i0 < total; i0 += 32) {
    const int i = i0 + lane;
    uint32_t item = 0;
    bool many = false;
    if (i < total) {
      item = list[i];
      const unsigned thr = step_threshold(item >> 14, neg);
      const uint32_t* const pa = Ah + unit_of<BS>((int)(item & 127u));
      const uint32_t* const pb = Bh + unit_of<BS>((int)(item >> 7 & 127u));
      uint32_t flags = scan_units<BS>(pa, pb, thr);
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
    }
    for (unsigned m = __ballot_sync(0xffffffffu, many); m; m &= m - 1) {
      const uint32_t got = __shfl_sync(0xffffffffu, item, __ffs((int)m) - 1);
      if (lane == naside) aside = got;
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
      const int k1 = item[u] >> 14 & 127u, k2 = item[u] >> 21 & 127u, n = item[u] >> 28;
      s1[u] = s2[u] = Num<T>::inf();
      best[u] = f.old[row * BS + col];
      if (n >= 1) s1[u] = operand<kGmem>(A + row * BS + k1) + operand<kGmem>(B + k1 * BS + col);
      if (n >= 2) s2[u] = operand<kGmem>(A + row * BS + k2) + operand<kGmem>(B + k2 * BS + col);
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
        store_relaxed(f, item[u] & 127u, item[u] >> 7 & 127u, best[u], arg[u], pred[u]);
  }
}

// Candidates of a warp from the minima of core_h (two halves per entry) and
// their exact relaxation.  list: one word per entry of the warp's part of the
// tile.  Whole warps.
template <typename T, int BS, bool kGmem>
__device__ __forceinline__ void refine_tile(const FilterTask<T>& f,
                                            const uint32_t (&acc)[Geo<BS>::TM][Geo<BS>::TM], int tx,
                                            int ty, uint32_t* list) {
  using Gm = Geo<BS>;
  constexpr int TM = Gm::TM, G = Gm::G;
  const int lane = threadIdx.x & 31;
  const QScale q = f.q;
  const int nrow = f.nrow, ncol = f.ncol;
  const bool neg = f.neg;
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
        const bool on = (neg || (F < kQInf && Quant<T>::may_improve(F, v[e], q))) && lr < nrow &&
                        lc + e < ncol;
        const unsigned all = __ballot_sync(0xffffffffu, on);
        if (on)
          list[total + __popc(all & below)] =
              at + ((uint32_t)Gm::idx(0, m) | (uint32_t)Gm::idx(0, g * G + e) << 7) + (F << 14);
        total += __popc(all);
      }
    }
  if (total == 0) return;
  __syncwarp();
  refine_list<T, BS, kGmem>(f, list, total);
  __syncwarp();
}

}  // namespace fwk
