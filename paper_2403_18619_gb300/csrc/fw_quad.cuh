// fp32 min-plus in groups of four steps.  The operands are stored step group
// by step group (units of four steps of one operand row, in the order of
// h_unit), so that an output takes four sums, two three-input minima and one
// update of its argmin -- the group that last lowered it -- per group: eight
// instructions for four relaxations, where an argmin by step takes sixteen.
// The step inside the group is found afterwards, for improved entries only, by
// summing the group's four steps again: the sums are the same IEEE sums, so the
// first one equal to their minimum is the step a relaxation in order with a
// strict compare would record.
//
// Measured from shared memory on GB300 (relaxations per SM clock): argmin by
// step 14-21, groups of two steps 23, of four 32-42 (fewer registers spilled),
// no argmin 60 (a two-input minimum per step: 49-57).
#pragma once

#include "fw_device.cuh"

namespace fwk {

__device__ __forceinline__ float min3f(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Shared-memory load that stays where it is written (loads hoisted above the
// work of earlier rows would spill the accumulators).
__device__ __forceinline__ float4 lds_here(const float* p) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(smem_u32(p)));
  return v;
}

// Relaxation over step groups g0 .. g0 + NGRP - 1, whose units start at As, Bs.
// arg: the last improving group of four entries per word, a byte each: the low
// six bits of a byte are those that the upper byte of 1.0f has set and that of
// 0.0f has not, so that the float compare's result selects them without a
// conversion.  (A float accumulator per entry, as in core_generic, or two
// entries per word leave too few registers under the kernel's 168-register
// cap: the loop spills, 31 relaxations per clock.)
template <int TM>
struct QuadArg {
  static constexpr int kWords = TM < 4 ? 1 : TM / 4;  // per micro-tile row
};
template <int BS, int NGRP, bool kArg>
__device__ __forceinline__ void core_q(const float* __restrict__ As, const float* __restrict__ Bs,
                                       float (&acc)[Geo<BS>::TM][Geo<BS>::TM],
                                       uint32_t (&arg)[Geo<BS>::TM][QuadArg<Geo<BS>::TM>::kWords],
                                       int tx, int ty, int g0) {
  // four columns at a time, for the same reason; a step's operands are loaded
  // during the step before it, a row's during the row before
  constexpr int TM = Geo<BS>::TM, NB = TM < 4 ? TM : 4, NH = TM / NB;
  static_assert(NH <= 2 && NGRP % 2 == 0, "two steps per pass of the loop");
  float4 b[2][NB], an;
#pragma unroll
  for (int nn = 0; nn < NB; ++nn) b[0][nn] = lds_here(Bs + h_unit<BS>(0, nn, tx));
  an = lds_here(As + h_unit<BS>(0, 0, ty));
#pragma unroll 1
  for (int s0 = 0; s0 < NGRP * NH; s0 += 2) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = s0 + h, g = s / NH, c0 = NH == 2 ? h * NB : 0;
      const int sx = min(s + 1, NGRP * NH - 1), gx = sx / NH, cx = NH == 2 ? (h ^ 1) * NB : 0;
      const uint32_t gg = (uint32_t)(g0 + g) * 0x01010101u;
#pragma unroll
      for (int m = 0; m < TM; ++m) {
        const float4 a = an;
        an = lds_here(As + (m + 1 < TM ? h_unit<BS>(g, m + 1, ty) : h_unit<BS>(gx, 0, ty)));
        if (m < NB) b[h ^ 1][m] = lds_here(Bs + h_unit<BS>(gx, cx + m, tx));
        uint32_t p[NB];
#pragma unroll
        for (int nn = 0; nn < NB; ++nn) {
          const float4& bb = b[h][nn];
          float& c = acc[m][c0 + nn];
          const float t = min3f(min3f(c, a.x + bb.x, a.y + bb.y), a.z + bb.z, a.w + bb.w);
          if (kArg) p[nn] = __float_as_uint(lt_one(t, c));
          c = t;
        }
        if (kArg) {
          uint32_t z = __byte_perm(p[0], p[1], 0x0073);
          if constexpr (NB == 4) z = __byte_perm(z, __byte_perm(p[2], p[3], 0x0073), 0x5410);
          uint32_t& r = arg[m][c0 / 4];
          r = (gg & z) | (r & ~z);
        }
      }
    }
  }
}

// Group of entry (m, nn) recorded by core_q.
template <int TM>
__device__ __forceinline__ uint32_t group_of(const uint32_t (&arg)[TM][QuadArg<TM>::kWords], int m,
                                             int nn) {
  return arg[m][nn / 4] >> (nn % 4 * 8) & 63u;
}

// First unit of operand row x = idx(t, m).
template <int BS>
__device__ __forceinline__ int unit_of(int x) {
  using Gm = Geo<BS>;
  return h_unit<BS>(0, (x / Gm::SPAN) * Gm::G + x % Gm::G, (x % Gm::SPAN) / Gm::G);
}

// One fp32 tile whose improved entries are to be stored.
struct QuadTask {
  const float* A;        // operands in step groups (shared memory, or global: kGmem)
  const float* B;
  const int32_t* Psrc;   // predecessors of B's rows, [kk][col] (BS < 128: shared memory)
  float* D;              // where the results go (kOutSmem: shared memory)
  int32_t* P;
  int64_t ld;
  bool diag;
  int* status;
};

// Step (0 .. 3) of a group whose sum is first equal to the group's minimum.
__device__ __forceinline__ int first_of(const float4& a, const float4& b) {
  const float s0 = a.x + b.x, s1 = a.y + b.y, s2 = a.z + b.z, s3 = a.w + b.w;
  const float best = min3f(fminf(s0, s1), s2, s3);
  return s0 == best ? 0 : s1 == best ? 1 : s2 == best ? 2 : 3;
}

// Entries of a warp's part of a tile in 16-bit list items: lane | nn << 5 |
// m << 8 | group << 11 (BS = 128: all 2048 of them in 4 KB).
template <int BS>
__device__ __forceinline__ void quad_entry(unsigned item, int& row, int& col, int& g) {
  using Gm = Geo<BS>;
  const int warp = threadIdx.x >> 5, l = item & 31u;
  row = Gm::idx((l >> 3) + 4 * (warp >> 1), item >> 8 & 7u);
  col = Gm::idx((l & 7) + 8 * (warp & 1), item >> 5 & 7u);
  g = (int)(item >> 11);
}

// Predecessors of `total` improved entries of one warp, four per lane at a time
// so that their loads overlap.
template <int BS, bool kGmem>
__device__ __noinline__ void finish_quads(const QuadTask& f, const uint16_t* list, int total) {
  constexpr int I = 4, kStride = Geo<BS>::TM * 64;
  const int lane = threadIdx.x & 31;
  const int64_t ld = f.ld;
  auto load = [](const float* p) -> float4 {
    if constexpr (kGmem) return __ldcg(reinterpret_cast<const float4*>(p));
    else return lds_here(p);
  };
#pragma unroll 1
  for (int i0 = lane; i0 < total; i0 += 32 * I) {
    int row[I], col[I], g[I];
    float4 a[I], b[I];
#pragma unroll
    for (int u = 0; u < I; ++u) {
      // (the last one again past the end)
      quad_entry<BS>(list[min(i0 + 32 * u, total - 1)], row[u], col[u], g[u]);
      a[u] = load(f.A + unit_of<BS>(row[u]) + g[u] * kStride);
      b[u] = load(f.B + unit_of<BS>(col[u]) + g[u] * kStride);
    }
    int32_t pred[I];
#pragma unroll
    for (int u = 0; u < I; ++u)
      pred[u] = __ldcg(f.Psrc + (g[u] * 4 + first_of(a[u], b[u])) * BS + col[u]);
#pragma unroll
    for (int u = 0; u < I; ++u)
      if (i0 + 32 * u < total) f.P[row[u] * ld + col[u]] = pred[u];
  }
}

// Stores what core_q improved against the tile's values `old` (shared memory,
// row-major): distances in vectors of the lanes' own entries, improved or not.
// Predecessors, BS = 128: by a list of the improved entries (an item per entry of
// the warp's part of the tile), since the operands come from global memory; small
// tiles, whose operands and predecessors are in shared memory: each lane its own.
// Whole warps.
template <int BS, bool kGmem, bool kOutSmem>
__device__ __forceinline__ void finish_tile_q(const QuadTask& f, const float* old, int nrow, int ncol,
                                              const float (&acc)[Geo<BS>::TM][Geo<BS>::TM],
                                              const uint32_t (&arg)[Geo<BS>::TM][QuadArg<Geo<BS>::TM>::kWords],
                                              int tx, int ty, uint16_t* list) {
  using Gm = Geo<BS>;
  constexpr int TM = Gm::TM, G = Gm::G, kStride = TM * 64;
  constexpr bool kList = BS == 128;
  const int lane = threadIdx.x & 31;
  const int64_t ld = f.ld;
  // the list entry by entry, all lanes' of one before the next, so that
  // neighbours in it lie in few row segments
  const unsigned below = (1u << lane) - 1u;
  int total = 0;
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lr = Gm::idx(ty, m), lc = g * Gm::SPAN + tx * G;
      float v[G];
      vload_s<G>(v, old + lr * BS + lc);
      bool better[G], any = false, neg = false;
      int32_t bits[G];
#pragma unroll
      for (int e = 0; e < G; ++e) {
        better[e] = acc[m][g * G + e] < v[e] && lr < nrow && lc + e < ncol;
        any |= better[e];
        v[e] = better[e] ? acc[m][g * G + e] : v[e];
        neg |= better[e] && f.diag && lr == lc + e && v[e] < 0.0f;
        bits[e] = __float_as_int(v[e]);
      }
      if constexpr (kOutSmem) {
        vstore<G>(f.D + lr * BS + lc, v);
      } else {
        int32_t* const Drow = reinterpret_cast<int32_t*>(f.D + lr * ld + lc);
        if (lc + G <= ncol) {
          st_if(any, Drow, bits);
        } else {
#pragma unroll
          for (int e = 0; e < G; ++e) st_if(any && lc + e < ncol, Drow + e, bits[e]);
        }
      }
      if (neg) atomicOr(f.status, kStNegCycle);
      if (!f.P) continue;
      if constexpr (kList) {
#pragma unroll
        for (int e = 0; e < G; ++e) {
          const int nn = g * G + e;
          const unsigned all = __ballot_sync(0xffffffffu, better[e]);
          if (better[e])
            list[total + __popc(all & below)] =
                (uint16_t)(lane | nn << 5 | m << 8 | group_of<TM>(arg, m, nn) << 11);
          total += __popc(all);
        }
      } else if (__any_sync(0xffffffffu, any)) {
        float4 a[G], b[G];
        int32_t pred[G];
        int kk[G];
        bool every = true;
#pragma unroll
        for (int e = 0; e < G; ++e) {
          const int nn = g * G + e;
          kk[e] = (int)group_of<TM>(arg, m, nn);
          a[e] = lds_here(f.A + h_unit<BS>(0, m, ty) + kk[e] * kStride);
          b[e] = lds_here(f.B + h_unit<BS>(0, nn, tx) + kk[e] * kStride);
          every &= better[e];
        }
#pragma unroll
        for (int e = 0; e < G; ++e)
          pred[e] = f.Psrc[(kk[e] * 4 + first_of(a[e], b[e])) * BS + lc + e];
        int32_t* const Prow = f.P + lr * ld + lc;
        if constexpr (kOutSmem) {
#pragma unroll
          for (int e = 0; e < G; ++e)
            if (better[e]) Prow[e] = pred[e];
        } else {
          st_if(every, Prow, pred);
#pragma unroll
          for (int e = 0; e < G; ++e) st_if(better[e] && !every, Prow + e, pred[e]);
        }
      }
    }
  if constexpr (kList) {
    if (total == 0) return;
    __syncwarp();
    finish_quads<BS, kGmem>(f, list, total);
    __syncwarp();
  }
}

}  // namespace fwk
