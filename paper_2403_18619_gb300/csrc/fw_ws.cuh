// Warp-specialised persistent driver (the GPU form of Opt-9's intra-round
// concurrency, Sec. 3.2, extended across rounds as the paper's future work
// proposes, Sec. 5).
//
// A CTA has 8 compute warps, 1 producer warp and 1 publisher warp.
//   * The producer claims tasks from a global queue in order, waits (bounded)
//     on the tiles' ready flags, and streams the operands of remaining-tile
//     tasks into shared memory with TMA copies while the compute warps work
//     on the previous task:
//       - the tile's own D block (one 2-D tensor copy, or one copy per row) -> Dbuf
//       - the A and B panel snapshots -> 2-stage ring: whole 16-bit tiles (keys
//         of int32, lower bounds of fp64), or chunks of 64 k-steps (64-bit
//         elements: 32) of values or 32-bit keys
//     and, for panel tasks, the tile and the closed pivot (ws_panel*).
//   * The compute warps relax and store improved entries; pivot tasks (and
//     panels of the 64-bit types where tiles are not filtered) are run by them
//     alone, using the shared buffer as scratch (the producer waits
//     until such a task is published).  The task that finishes tile
//     (r+1, r+1) of round r runs the pivot of round r+1 right after it.
//   * The publisher sleeps on the compute warps' task-done barrier and
//     publishes each finished tile (the GPU-scope release), so that neither the
//     compute warps nor the producer wait on that fence.
// mbarriers carry "full" (transaction bytes landed) and "empty" (readers done)
// signals.
//
// The same engine runs one graph (fw_solve) or a batch of graphs with
// different sizes and block sizes in one launch (fw_solve_batched): a "task
// source" maps a global queue index to (graph, task).
#pragma once

#include "fw_device.cuh"
#include "fw_filter.cuh"
#include "fw_quad.cuh"
#include "fw_internal.h"

namespace fwk {

// 10 warps: 8 compute, 1 producer, 1 publisher.  Three of them share one SM
// sub-partition, whose 16K registers then cap the kernel at 168 registers per
// thread (ptxas derives this from the launch bounds).  (Four more warps that
// did the epilogue of a 16-bit tile while the compute warps relaxed the next
// starved: the relaxations hold the ALU pipe, n = 16384 300 ms against 180.)
constexpr int kWsThreads = kThreads + 64;
constexpr int kPubDepth = 4;  // tasks handed to the compute warps but not yet published
// Internal task type: remaining tile (r+1, r+1) of round r followed, on the
// same CTA and without a publication in between, by the pivot of round r+1
// (whose own queue entry is then skipped).  That tile is the pivot's only
// input, so the pivot starts as soon as the tile is relaxed: one hand-off
// less on the chain that bounds small solves (pivot -> panels -> tile ->
// next pivot).
constexpr int kFusedTask = 4;

// The exact 64-bit kernels run panels by the compute warps alone (task_panel).
template <typename T, int BS>
constexpr bool kOwnPanels = sizeof(T) == 8 && !kFiltered<T, BS>;

// Floating types, small tiles: the predecessors that improved entries take come
// into the ring stage, beside the operands, and stay there until the epilogue is
// done with them.  fp32 keeps its operands as well: the epilogue's chain of loads
// (a group's operands, then the predecessor) from global memory cost more than
// the relaxation (a tile of 64: relaxed in 5.6 K cycles, done after 17 K; now
// 8.3 and 13.4); fp64 in tiles of 32: 23.6 K cycles, now 22.1.  A ring for tiles
// of 128 has no room.
template <typename T, int BS>
constexpr bool kPredSmem = std::is_same<T, float>::value ? BS <= 64
                                                         : std::is_same<T, double>::value && BS <= 32;

// Operand chunks of a task that streams values or 32-bit keys: CK k-steps of A
// and of B, 64 at most (64-bit elements: 32), so that a BS = 128 task takes two.
template <int BS, typename T>
struct WsChunk {
  static constexpr int kMax = sizeof(T) == 4 ? 64 : 32;
  static constexpr int CK = BS < kMax ? BS : kMax;                        // k-steps per chunk
  static constexpr int NC = BS / CK;                                      // chunks per task
  static constexpr size_t kChunkBytes = (size_t)CK * BS * sizeof(T);      // one operand chunk
  static constexpr size_t kTile = (size_t)BS * BS * sizeof(T);            // a tile of elements
  static constexpr size_t kHTile = (size_t)BS * BS * 2;                   // a 16-bit tile
};

// Shared-memory layout sized for the largest block size LBS a launch runs:
// the 2-stage operand ring (a stage holds two 16-bit tiles, a tile of elements
// or two 32-bit chunks), the tile's own D (Dbuf) and, where an epilogue lists the
// improved entries, an item per entry (fp32 tiles of 128: 2 bytes; filtered fp64
// tiles: 4).  LBS = 128: fp32 224 KB, int32 192 KB (which leaves 60 KB of L1 cache
// instead of 28: n = 8000 1.3 % faster); fp64 of 64: 112 KB, two CTAs per SM.
template <int LBS, typename T>
struct WsLayout {
  static constexpr size_t kTile = WsChunk<LBS, T>::kTile;
  static constexpr size_t kHTile = WsChunk<LBS, T>::kHTile;
  static constexpr size_t kStage =
      2 * WsChunk<LBS, T>::kChunkBytes + (kPredSmem<T, LBS> ? (size_t)LBS * LBS * 4 : 0);
  static constexpr size_t kRing = 2 * kStage;
  static constexpr size_t kScr = kFiltered<T, LBS>                                ? (size_t)LBS * LBS * 4
                                 : std::is_same<T, float>::value && LBS == 128 ? kHTile
                                                                               : 0;
  static constexpr size_t kScrWarp = kScr / (kThreads / 32);
  __host__ __device__ static constexpr size_t ring_off() { return 0; }
  __host__ __device__ static constexpr size_t d_off() { return kRing; }
  __host__ __device__ static constexpr size_t scr_off() { return kRing + kTile; }
  __host__ __device__ static constexpr size_t bytes() { return scr_off() + kScr; }
  static_assert(2 * kHTile <= kStage && kTile <= kStage, "a stage holds either");
  // the int32 pivot uses the buffer from offset 0 as three tiles of scratch,
  // task_panel as two tiles and one of predecessors
  static_assert(!Num<T>::kPacked || bytes() >= 3 * kTile, "scratch of pivot tasks");
  static_assert(!kOwnPanels<T, LBS> || bytes() >= 2 * kTile + (size_t)LBS * LBS * 4, "task_panel");
  static_assert(bytes() <= 226 * 1024, "shared memory of one CTA");
};

struct WsBars {
  uint64_t desc_full[2], desc_empty[2];
  uint64_t chunk_full[2], chunk_empty[2];
  uint64_t d_full, d_empty;
  // one completion barrier per publication slot: the compute warps may finish
  // several tasks while one publication is under way, and a parity wait only
  // tells the latest two phases apart
  uint64_t task_done[kPubDepth];
  uint64_t pub_full[kPubDepth], pub_empty[kPubDepth];
  int desc[2][8];           // t, type, r, ti, tj, mode, graph, key operands
  int pubq[kPubDepth][6];   // t, type, r, ti, tj, graph of tasks awaiting publication
  int pst[kPubDepth];       // what the publisher stores for the task (kPst*; ws_panel_h)
};

// A 16-bit panel task leaves its results in shared memory and the publisher
// stores them (store_panel): the ring stage of the live tile (the other one
// holds the 16-bit snapshot), and whether the tile is whole and stored so.
constexpr int kPstOn = 1, kPstStage = 2, kPstTile = 4;

// Wait on an mbarrier phase of this CTA.  Such a phase ends by the CTA's own
// progress: a descriptor that the producer hands out (the last one says stop), a
// copy that it issues after the task's inputs from other CTAs are there, a buffer
// that the warps leave.  Only the producer waits for other CTAs (wait_ge), and only
// there the solve's limit and its abort flag count: the producer alone decides that
// a solve ends early, and every warp learns of it by the same descriptor.  (With a
// limit here, warps would give up one by one, and those that did not would be left
// at a barrier: a turn, or the barriers of pivots and panels.)
// False, with the timeout status, only if the phase is still open kLostNs after
// the longest wait of the producer: a copy was lost.
constexpr uint64_t kLostNs = 10000000000ull;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int* status,
                                          int* abort_flag, int64_t timeout_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (int64_t it = 0; it < ((int64_t)1 << 30); ++it) {
    if (mbar_try_wait_sleep(bar, parity, 20000u)) return true;
    if ((it & 15) == 15 && globaltimer() - t0 > (uint64_t)timeout_ns + kLostNs) break;
  }
  atomicOr(status, kStTimeout);
  atomicExch(abort_flag, 1);
  return false;
}

// A cycle count clamped to 20 bits (three of them share a trace word).
__device__ __forceinline__ uint64_t cyc20(long long c) {
  return (uint64_t)(c < 0 ? 0 : c > 0xfffff ? 0xfffff : c);
}

// Scalars the compute warps need, passed by value (kept in registers).
template <typename T>
struct TileCtx {
  T* D;
  int32_t* P;
  int64_t n, ld;
  int r;                // round
  int* status;
  int* abort_flag;
  int64_t timeout_ns;
};

// Counters of the shared-memory pipelines (each side keeps its own copy).
// The producer also records, per full barrier, 1 + the last phase it armed
// with a copy (0: none), and stops arming once a wait has given up: arming a
// phase whose predecessor has not completed would add its bytes to the wrong
// phase.
// (The drain waits on the LAST phase of each barrier: a parity wait can only
// tell the latest two phases apart.)
struct PipeCnt {
  unsigned d = 0, chunk = 0;
  unsigned d_armed = 0, chunk_armed[2] = {0, 0};
  bool stop = false;
  int exact = -2;  // (filtered fp64) skip_filter
};

// ------------------------------------------------------------ compute side ----

// Operand forms of a remaining tile (tile_form).
constexpr int kFormKA = 1, kFormKB = 2, kFormHA = 4, kFormHB = 8, kFormInfA = 16, kFormInfB = 32;

// In-place decode of `count` packed keys (int32 path) back to values, for a
// remaining tile relaxed with compare and select whose panel wrote its key
// snapshot only (exact: every finite value was below CAP).  Compute warps
// only; the caller synchronises them before reading the buffer.
template <int BS>
__device__ __forceinline__ void decode_keys(uint32_t* buf, int count) {
  using K = Keys<BS>;
  for (int i = (int)threadIdx.x * 4; i < count; i += kThreads * 4) {
    uint4 v = *reinterpret_cast<uint4*>(buf + i);
    auto d = [](uint32_t k) -> uint32_t {
      const uint32_t x = k >> K::KB;
      return x == (uint32_t)K::CAP ? (uint32_t)Num<int32_t>::inf() : x;
    };
    v.x = d(v.x);
    v.y = d(v.y);
    v.z = d(v.z);
    v.w = d(v.w);
    *reinterpret_cast<uint4*>(buf + i) = v;
  }
}

// Expansion of a 16-bit snapshot tile at buf, in place, to the chunk of CK
// steps from step ch * CK: 32-bit keys (with the code of the step for an A
// operand) or values.  The tile goes through registers, so that no word is
// overwritten before it is read.
template <int BS, int CK>
__device__ __noinline__ void expand_h(uint32_t* buf, int ch, bool keys, bool is_a, bool has_inf) {
  using H = KeysH<BS>;
  using K = Keys<BS>;
  using Gm = Geo<BS>;
  constexpr int TM = Gm::TM;
  uint32_t words[H::kTileWords / kThreads];
#pragma unroll
  for (int j = 0; j < H::kTileWords / kThreads; ++j) words[j] = buf[threadIdx.x + j * kThreads];
  bar_compute();
#pragma unroll
  for (int j = 0; j < H::kTileWords / kThreads; ++j) {
    const int i = (int)threadIdx.x + j * kThreads;
    const uint32_t w = words[j];
    const int row = Gm::idx((i >> 2) & 15, (i >> 6) % TM), kw = (i >> 6) / TM * 4 + (i & 3);
    auto put = [&](int h) {
      const int kk = kk_of<BS>(kw, h);
      const int d = (int)((w >> (16 * h)) & 0xffffu) >> H::KB;
      const bool inf = has_inf && d == H::kCapI;
      buf[(kk - ch * CK) * BS + row] =
          keys ? ((uint32_t)(inf ? K::CAP : d) << K::KB) + (is_a ? (uint32_t)kk + 1u : 0u)
               : (uint32_t)(inf ? Num<int32_t>::inf() : d);
    };
    if constexpr (CK == BS) {
      put(0);
      put(1);
    } else {
      static_assert(CK == BS || (BS == 128 && CK == 64), "a half of the words per chunk");
      put(ch);
    }
  }
}

// Operands of a remaining tile that arrive in another form than its core reads
// (tile_form): 32-bit keys decoded to values, a 16-bit snapshot expanded,
// in the ring stage (every warp has waited for the stage to fill, so no warp
// still reads its previous contents); synchronises the compute warps.
template <typename T, int BS, int CK>
__device__ __forceinline__ void decode_chunk(unsigned char* stage, int dec, int ch, bool keys) {
  if constexpr (Num<T>::kPacked) {
    if (!(dec & (kFormKA | kFormKB | kFormHA | kFormHB))) return;
    uint32_t* As = reinterpret_cast<uint32_t*>(stage);
    if (dec & kFormKA) decode_keys<BS>(As, CK * BS);
    if (dec & kFormKB) decode_keys<BS>(As + CK * BS, CK * BS);
    if (dec & kFormHA) expand_h<BS, CK>(As, ch, keys, true, dec & kFormInfA);
    if (dec & kFormHB) expand_h<BS, CK>(As + CK * BS, ch, keys, false, dec & kFormInfB);
    fence_proxy_async_shared();  // generic writes before the stage's next TMA fill
    bar_compute();
  }
}

// Distance-only remaining-tile task (no predecessors, generic kernel): add +
// min over the streamed chunks, then the whole tile written back (unchanged
// entries rewrite their own value).  A function of its own, so that the
// packed kernel's register allocation does not see it.
template <typename T, int BS, int LBS>
__device__ __noinline__ bool ws_minplus_dist(TileCtx<T> c, int ti, int tj, int dec,
                                             unsigned char* smem, WsBars* wb, PipeCnt& pc,
                                             uint64_t* tr) {
  using Gm = Geo<BS>;
  using L = WsLayout<LBS, T>;
  using C = WsChunk<BS, T>;
  constexpr int TM = Gm::TM, G = Gm::G;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const T* Dbuf = reinterpret_cast<const T*>(smem + L::d_off());
  unsigned char* ring = smem + L::ring_off();
  const int64_t row0 = (int64_t)ti * BS, col0 = (int64_t)tj * BS;
  const int nrow = (int)(c.n - row0 < BS ? c.n - row0 : BS);
  const int ncol = (int)(c.n - col0 < BS ? c.n - col0 : BS);
  const bool full = nrow == BS && ncol == BS;
  const long long t_a = tr ? clock64() : 0;
  long long cw = 0;
  if (!mbar_wait(&wb->d_full, pc.d & 1, c.status, c.abort_flag, c.timeout_ns)) return false;
  const long long t_b = tr ? clock64() : 0;
  T acc[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lc0 = g * Gm::SPAN + tx * G;
      T tmp[G];
      vload_s<G>(tmp, Dbuf + lr * BS + lc0);
#pragma unroll
      for (int e = 0; e < G; ++e)
        acc[m][g * G + e] = (lr < nrow && lc0 + e < ncol) ? tmp[e] : Num<T>::inf();
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(&wb->d_empty);
  ++pc.d;
  for (int ch = 0; ch < C::NC; ++ch) {
    const unsigned st = pc.chunk & 1;
    const long long w0 = tr ? clock64() : 0;
    if (!mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, c.status, c.abort_flag,
                   c.timeout_ns))
      return false;
    if (tr) cw += clock64() - w0;
    decode_chunk<T, BS, C::CK>(ring + st * L::kStage, dec, ch, false);
    const T* As = reinterpret_cast<const T*>(ring + st * L::kStage);
    const T* Bs = As + C::CK * BS;
    core_min<BS, T, C::CK>(As, Bs, acc, tx, ty);
    __syncwarp();
    if (lane == 0) mbar_arrive(&wb->chunk_empty[st]);
    ++pc.chunk;
  }
  if (tr) {
    tr[7] = cyc20(t_b - t_a) | (cyc20(cw) << 20);
    tr[8] = (uint64_t)(clock64() - t_a);
  }
  T* Drow = c.D + row0 * c.ld + col0;
  bool neg = false;
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lc0 = g * Gm::SPAN + tx * G;
      T v[G];
#pragma unroll
      for (int e = 0; e < G; ++e) {
        v[e] = acc[m][g * G + e];
        neg |= (row0 + lr == col0 + lc0 + e) && v[e] < T(0);
      }
      if (full) {
        vstore<G>(Drow + lr * c.ld + lc0, v);
      } else if (lr < nrow) {
#pragma unroll
        for (int e = 0; e < G; ++e)
          if (lc0 + e < ncol) Drow[lr * c.ld + lc0 + e] = v[e];
      }
    }
  }
  if (tr) tr[8] |= (uint64_t)(clock64() - t_a) << 32;
  if (neg) atomicOr(c.status, kStNegCycle);
  return true;
}

// Turns of the two groups of compute warps (0-3 and 4-7, one warp of each per
// SM sub-partition) in the relaxation of a 16-bit tile: one group relaxes at
// the full rate of the ALU pipe while the other stores what its previous turn
// improved, which is bound by latency and the load/store unit (8 K SM cycles
// per tile, whatever the layout; both groups in step 27 K cycles per tile,
// 19 K of them relaxation).  Named barriers 2 + g: group g may go.
__device__ __forceinline__ void turn_wait(int g) {
  if (g) asm volatile("bar.sync 3, 256;" ::: "memory");
  else asm volatile("bar.sync 2, 256;" ::: "memory");
}
__device__ __forceinline__ void turn_pass(int g) {
  if (g) asm volatile("bar.arrive 3, 256;" ::: "memory");
  else asm volatile("bar.arrive 2, 256;" ::: "memory");
}

// Remaining-tile task over 16-bit packed keys (int32; cap: their clamp).  The
// accumulators hold the operands' sums only; the tile's own values are read
// from Dbuf afterwards, so that their copy has the whole relaxation to arrive
// and nothing converts them to keys.  Bound by the ALU pipe (two relaxations per
// DPX instruction, 122 per SM clock), which the turns keep to the relaxation:
// n = 16384 265 ms over 32-bit keys, 174 ms.
template <typename T, int BS, int LBS>
__device__ __noinline__ bool ws_minplus_h(const Args<T>& a, const fwh::Task& k, int cap,
                                          unsigned char* smem, WsBars* wb, PipeCnt& pc,
                                          uint64_t* tr) {
  using Gm = Geo<BS>;
  using H = KeysH<BS>;
  using L = WsLayout<LBS, T>;
  constexpr int TM = Gm::TM, G = Gm::G;
  const int lane = threadIdx.x & 31;
  int tx, ty;
  h_thread(tx, ty);
  const T* const Dbuf = reinterpret_cast<const T*>(smem + L::d_off());
  const unsigned st = pc.chunk & 1;
  const long long t_a = tr ? clock64() : 0;
  if (!mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, a.status, a.abort_flag, a.timeout_ns))
    return false;
  const long long cw = tr ? clock64() - t_a : 0;
  uint32_t acc[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) acc[m][nn] = 0xffffffffu;
  const int group = (int)threadIdx.x >> 7;
  turn_wait(group);
  const uint32_t* const As = reinterpret_cast<const uint32_t*>(smem + L::ring_off() + st * L::kStage);
  core_h<BS>(As, As + H::kTileWords, acc, tx, ty);
  turn_pass(group ^ 1);
  __syncwarp();
  if (lane == 0) mbar_arrive(&wb->chunk_empty[st]);
  ++pc.chunk;
  const long long t_b = tr ? clock64() : 0;
  if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns)) return false;
  if (tr) {
    tr[7] = cyc20(clock64() - t_b) | (cyc20(cw) << 20);
    tr[8] = (uint64_t)(t_b - t_a);
  }
  const int64_t ld = a.ld, row0 = (int64_t)k.ti * BS, col0 = (int64_t)k.tj * BS;
  const int nrow = (int)(a.n - row0 < BS ? a.n - row0 : BS);
  const int ncol = (int)(a.n - col0 < BS ? a.n - col0 : BS);
  const bool whole = nrow == BS && ncol == BS;
  T* const D = a.D + row0 * ld + col0;
  int32_t* const P = a.P ? a.P + row0 * ld + col0 : nullptr;
  const int32_t via0 = via_code((int64_t)k.r * BS);  // via_code(k) = via0 - kk
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
    T* const Drow = D + lr * ld;
    int32_t* const Prow = P + lr * ld;
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lc = g * Gm::SPAN + tx * G;
      T v[G];
      vload_s<G>(v, Dbuf + lr * BS + lc);
      int kk[G];
      bool better[G], any = false;
#pragma unroll
      for (int e = 0; e < G; e += 2) {
        const uint32_t mm = h_min2(acc[m][g * G + e], acc[m][g * G + e + 1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int d = h ? (int)(mm >> (16 + H::KB)) : (int)((mm >> H::KB) & (H::kCapF));
          kk[e + h] = (int)((h ? mm >> 16 : mm) & H::MASK);
          // (sums with an INF operand are at or above the clamp)
          better[e + h] = d < (int)v[e + h] && d < cap && lr < nrow && lc + e + h < ncol;
          if (better[e + h]) v[e + h] = (T)d;
          any |= better[e + h];
        }
      }
      if (whole) {
        st_if(any, Drow + lc, v);
      } else {
#pragma unroll
        for (int e = 0; e < G; ++e) st_if(better[e], Drow + lc + e, v[e]);
      }
      if (P) {
#pragma unroll
        for (int e = 0; e < G; ++e) st_if(better[e], Prow + lc + e, via0 - kk[e]);
      }
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(&wb->d_empty);
  ++pc.d;
  if (tr) tr[8] |= (uint64_t)(clock64() - t_a) << 32;
  return true;
}

// fp32: the parts of a QuadTask that follow from the tile (ti, tj).
template <int BS>
__device__ __forceinline__ QuadTask quad_task(const Args<float>& a, int ti, int tj) {
  QuadTask f;
  f.D = a.D + (int64_t)ti * BS * a.ld + (int64_t)tj * BS;
  f.P = a.P ? a.P + (int64_t)ti * BS * a.ld + (int64_t)tj * BS : nullptr;
  f.ld = a.ld;
  f.diag = ti == tj;
  f.status = a.status;
  return f;
}

// Remaining-tile task of fp32, bound by issue slots (eight instructions per four
// relaxations).  Tiles of 128 with predecessors are relaxed in turns, each group of
// warps with the pipes to itself while the other finds the steps of what it
// improved (n = 8192: 78 ms, 83 without turns; 73 since distances leave in
// vectors, 71 in a function of its own, 98 with an argmin by step); distances alone leave little to do
// afterwards (n = 5000: 10.5 ms without turns, 11.9 with), and small tiles wait on
// a chain, which turns lengthen (a tile of 64: 17 K SM cycles, 13.4 K without).
// A function each for tiles with predecessors (kPred) and without: as one, the tile of
// 128 reloads 264 bytes of spilled registers, apart 224 with predecessors and 8 without
// (n = 5000 without predecessors 10.7 -> 9.8 ms, with them 18.0 -> 17.5).  Tiles of 64
// spill in neither form and gain too (n = 2900 without 2.62 -> 2.34); why is not known.
template <int BS, int LBS, bool kPred>
__device__ __noinline__ bool ws_minplus_q(const Args<float>& a, const fwh::Task& k,
                                          unsigned char* smem, WsBars* wb, PipeCnt& pc,
                                          uint64_t* tr) {
  using L = WsLayout<LBS, float>;
  using C = WsChunk<BS, float>;
  constexpr int TM = Geo<BS>::TM;
  const int lane = threadIdx.x & 31;
  int tx, ty;
  h_thread(tx, ty);
  const long long t_a = tr ? clock64() : 0;
  long long cw = 0;
  float acc[TM][TM];
  uint32_t arg[TM][QuadArg<TM>::kWords];
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) {
      acc[m][nn] = Num<float>::inf();
      arg[m][nn / 4] = 0;
    }
  constexpr bool kHold = kPredSmem<float, BS>;  // the operands stay for the epilogue
  constexpr bool kTurns = !kHold && kPred;
  static_assert(!kHold || C::NC == 1, "all of a tile's operands in one stage");
  const unsigned st0 = pc.chunk & 1;
  unsigned char* const stage0 = smem + L::ring_off() + st0 * L::kStage;
  const int group = (int)threadIdx.x >> 7;
  bool ok = mbar_wait(&wb->chunk_full[pc.chunk & 1], (pc.chunk >> 1) & 1, a.status, a.abort_flag,
                      a.timeout_ns);
  if (kTurns) turn_wait(group);
#pragma unroll 1
  for (int ch = 0; ch < C::NC && ok; ++ch) {
    const unsigned st = pc.chunk & 1;
    const long long w0 = tr ? clock64() : 0;
    ok = mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, a.status, a.abort_flag, a.timeout_ns);
    if (!ok) break;
    if (tr) cw += clock64() - w0;
    const float* const As = reinterpret_cast<const float*>(smem + L::ring_off() + st * L::kStage);
    const float* const Bs = As + C::CK * BS;
    core_q<BS, C::CK / 4, kPred>(As, Bs, acc, arg, tx, ty, kPred ? ch * (C::CK / 4) : 0);
    __syncwarp();
    if (!kHold && lane == 0) mbar_arrive(&wb->chunk_empty[st]);
    ++pc.chunk;
  }
  if (kTurns) turn_pass(group ^ 1);
  if (!ok) return false;
  const long long t_b = tr ? clock64() : 0;
  if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns)) return false;
  if (tr) {
    tr[7] = cyc20(clock64() - t_b) | (cyc20(cw) << 20);
    tr[8] = (uint64_t)(t_b - t_a);
  }
  QuadTask f = quad_task<BS>(a, k.ti, k.tj);
  if (!kPred) f.P = nullptr;
  const size_t ta = (size_t)(k.r & 1) * a.slot_tiles + k.ti, tb = (size_t)(k.r & 1) * a.slot_tiles + k.tj;
  if constexpr (kHold) {
    f.A = reinterpret_cast<const float*>(stage0);
    f.B = f.A + BS * BS;
    f.Psrc = reinterpret_cast<const int32_t*>(f.B + BS * BS);
  } else {
    f.A = a.colR + ta * BS * BS;
    f.B = a.rowR + tb * BS * BS;
    f.Psrc = a.rowP + tb * BS * BS;
  }
  const int64_t row0 = (int64_t)k.ti * BS, col0 = (int64_t)k.tj * BS;
  finish_tile_q<BS, !kHold, false>(f, reinterpret_cast<const float*>(smem + L::d_off()),
                          (int)(a.n - row0 < BS ? a.n - row0 : BS),
                          (int)(a.n - col0 < BS ? a.n - col0 : BS), acc, arg, tx, ty,
                          reinterpret_cast<uint16_t*>(smem + L::scr_off() +
                                                      (threadIdx.x >> 5) * L::kScrWarp));
  __syncwarp();
  if (lane == 0) {
    mbar_arrive(&wb->d_empty);
    if (kHold) mbar_arrive(&wb->chunk_empty[st0]);
  }
  ++pc.d;
  if (tr) tr[8] |= (uint64_t)(clock64() - t_a) << 32;
  return true;
}

// Unit of a BS x BS tile for thread slot i (0 .. BS*BS/4 - 1): operand row x and
// step group g.  kA: steps along the tile's columns; a warp takes 8 operand rows
// times 4 groups, so that it reads 64 bytes of each row and writes whole lines.
// Else steps along the rows; a warp takes 32 operand rows (columns of the tile).
template <int BS, bool kA>
__device__ __forceinline__ void unit_at(int i, int& x, int& g) {
  if constexpr (kA) {
    const int l = i & 31, w = i >> 5, rest = w / (BS / 16);
    g = (l & 3) + 4 * (w % (BS / 16));
    x = Geo<BS>::idx((l >> 2) + 8 * (rest & 1), rest >> 1);
  } else {
    x = i % BS;
    g = i / BS;
  }
}

// Panel task of fp32: Dbuf holds the tile's own values and ring stage s0 the
// closed pivot; both are rewritten in step groups, the own values into stage s1,
// the pivot in place.  Small tiles (kPredSmem) are relaxed within shared memory:
// s0 and s1 hold the predecessors as well, and the result leaves in whole rows.
// (By way of the matrix and with the predecessors in global memory a row panel
// of 64 took 24.5 K cycles, 10 K of them after the relaxation.)  A tile of 128
// stores its improved entries to the matrix and makes its snapshots (step
// groups, a row tile's predecessors) from there; a row tile's old predecessors
// wait in the snapshot's place meanwhile.
template <int BS, int LBS, bool is_row>
__device__ __noinline__ bool ws_panel_q(const Args<float>& a, const fwh::Task& k,
                                        unsigned char* smem, WsBars* wb, PipeCnt& pc) {
  using L = WsLayout<LBS, float>;
  constexpr int TM = Geo<BS>::TM;
  constexpr bool kSmem = kPredSmem<float, BS>;
  static_assert(!kSmem || 3 * WsChunk<BS, float>::kTile <= L::kStage, "three tiles per stage");
  const int tid = threadIdx.x, lane = tid & 31;
  int tx, ty;
  h_thread(tx, ty);
  const int r = k.r, t = is_row ? k.tj : k.ti;
  const unsigned s0 = pc.chunk & 1, s1 = s0 ^ 1;
  float* const own = reinterpret_cast<float*>(smem + L::d_off());
  float* const pivq = reinterpret_cast<float*>(smem + L::ring_off() + s0 * L::kStage);
  float* const ownq = reinterpret_cast<float*>(smem + L::ring_off() + s1 * L::kStage);
  // (kSmem) the own predecessors before and after, one tile each
  int32_t* const predOld = reinterpret_cast<int32_t*>(ownq + BS * BS);
  int32_t* const predNew = predOld + BS * BS;
  stamp(0);
  QuadTask f = quad_task<BS>(a, k.ti, k.tj);
  float* const Dt = f.D;
  int32_t* const Pt = f.P;
  const int64_t ld = a.ld;
  const int64_t row0 = (int64_t)k.ti * BS, col0 = (int64_t)k.tj * BS;
  const int nrow = (int)(a.n - row0 < BS ? a.n - row0 : BS);
  const int ncol = (int)(a.n - col0 < BS ? a.n - col0 : BS);
  const size_t tile = (size_t)(r & 1) * a.slot_tiles + t;
  int32_t* const snapP = a.rowP + tile * BS * BS;
  if (!mbar_wait(&wb->chunk_full[s1], ((pc.chunk + 1) >> 1) & 1, a.status, a.abort_flag,
                 a.timeout_ns))
    return false;
  if (Pt) {
    if constexpr (kSmem) {
      stage_tile_i32<BS>(predNew, a.P, a.n, a.ld, k.ti, k.tj, nullptr);
      if constexpr (is_row) {
        for (int q = tid; q < BS * BS / 4; q += kThreads)
          reinterpret_cast<int4*>(predOld)[q] = reinterpret_cast<const int4*>(predNew)[q];
      }
    } else if constexpr (is_row) {
      stage_tile_i32<BS>(snapP, a.P, a.n, a.ld, k.ti, k.tj, nullptr);
    }
  }
  if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns) ||
      !mbar_wait(&wb->chunk_full[s0], (pc.chunk >> 1) & 1, a.status, a.abort_flag,
                 a.timeout_ns))
    return false;
  constexpr int NU = BS * BS / 4 / kThreads;  // units per thread
  float4 pv[NU];
#pragma unroll
  for (int j = 0; j < NU; ++j) {
    int x, g;
    unit_at<BS, is_row>(tid + j * kThreads, x, g);
    if constexpr (is_row) {
      pv[j] = *reinterpret_cast<const float4*>(pivq + x * BS + 4 * g);
    } else {
      const float* const p = pivq + 4 * g * BS + x;
      pv[j] = make_float4(p[0], p[BS], p[2 * BS], p[3 * BS]);
    }
  }
  // the own values as an operand (entries beyond n: INF)
  auto own_unit = [&](int j, auto&& at) -> float4 {
    int x, g;
    unit_at<BS, !is_row>(tid + j * kThreads, x, g);
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int lr = is_row ? 4 * g + e : x, lc = is_row ? x : 4 * g + e;
      v[e] = lr < nrow && lc < ncol ? at(lr, lc) : Num<float>::inf();
    }
    return make_float4(v[0], v[1], v[2], v[3]);
  };
  auto unit_off = [&](int j, auto kA) -> int {
    int x, g;
    unit_at<BS, decltype(kA)::value>(tid + j * kThreads, x, g);
    return unit_of<BS>(x) + g * TM * 64;
  };
  using Row = std::integral_constant<bool, is_row>;
  using Col = std::integral_constant<bool, !is_row>;
  auto own_at = [&](int lr, int lc) { return own[lr * BS + lc]; };
#pragma unroll
  for (int j = 0; j < NU; ++j)
    *reinterpret_cast<float4*>(ownq + unit_off(j, Col{})) = own_unit(j, own_at);
  bar_compute();  // the pivot is in registers
#pragma unroll
  for (int j = 0; j < NU; ++j) *reinterpret_cast<float4*>(pivq + unit_off(j, Row{})) = pv[j];
  bar_compute();  // (and the old predecessors are in place)
  stamp(1);
  float acc[TM][TM];
  uint32_t arg[TM][QuadArg<TM>::kWords];
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) {
      acc[m][nn] = Num<float>::inf();
      arg[m][nn / 4] = 0;
    }
  f.A = is_row ? pivq : ownq;
  f.B = is_row ? ownq : pivq;
  if constexpr (kSmem) {
    f.D = own;
    f.P = Pt ? predNew : nullptr;
    f.ld = BS;
    f.Psrc = is_row ? predOld : reinterpret_cast<const int32_t*>(pivq + BS * BS);
  } else {
    f.Psrc = is_row ? snapP : a.pivP + (size_t)(r & 1) * BS * BS;
  }
  // (No argmin that nobody reads: without predecessors n = 5000 9.8 -> 9.5 ms, n = 2048
  // 1.13 -> 1.10, n = 2900 2.33 -> 2.33.)
  if (Pt) core_q<BS, BS / 4, true>(f.A, f.B, acc, arg, tx, ty, 0);
  else core_q<BS, BS / 4, false>(f.A, f.B, acc, arg, tx, ty, 0);
  finish_tile_q<BS, false, kSmem>(f, own, nrow, ncol, acc, arg, tx, ty,
                                         reinterpret_cast<uint16_t*>(smem + L::scr_off() +
                                                                     (tid >> 5) * L::kScrWarp));
  if constexpr (!kSmem) fence_proxy_async_shared();  // generic writes before the next TMA fill
  bar_compute();  // the relaxed tile is complete (kSmem: in own, else in the matrix)
  stamp(2);
  auto release = [&] {
    if (lane == 0) {
      mbar_arrive(&wb->d_empty);
      mbar_arrive(&wb->chunk_empty[0]);
      mbar_arrive(&wb->chunk_empty[1]);
    }
  };
  float* const snapR = (is_row ? a.rowR : a.colR) + tile * BS * BS;
  if constexpr (kSmem) {
#pragma unroll
    for (int j = 0; j < NU; ++j) {
      const int q = tid + j * kThreads, lr = q / (BS / 4), lc = q % (BS / 4) * 4;
      const float4 v = *reinterpret_cast<const float4*>(own + lr * BS + lc);
      int4 p = make_int4(-1, -1, -1, -1);
      if (Pt) {
        p = *reinterpret_cast<const int4*>(predNew + lr * BS + lc);
        if constexpr (is_row) *reinterpret_cast<int4*>(snapP + lr * BS + lc) = p;
      }
      if (lr < nrow && lc + 4 <= ncol) {
        *reinterpret_cast<float4*>(Dt + lr * ld + lc) = v;
        if (Pt) *reinterpret_cast<int4*>(Pt + lr * ld + lc) = p;
      } else if (lr < nrow) {
        const float ve[4] = {v.x, v.y, v.z, v.w};
        const int32_t pe[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (lc + e < ncol) {
            Dt[lr * ld + lc + e] = ve[e];
            if (Pt) Pt[lr * ld + lc + e] = pe[e];
          }
      }
    }
#pragma unroll
    for (int j = 0; j < NU; ++j)
      *reinterpret_cast<float4*>(snapR + unit_off(j, Col{})) = own_unit(j, own_at);
    fence_proxy_async_shared();  // generic writes before the buffers' next TMA fill
    __syncwarp();
    release();
  } else {
    release();
    if (is_row && Pt) stage_tile_i32<BS>(snapP, a.P, a.n, a.ld, k.ti, k.tj, nullptr);
    constexpr int kAhead = 4;  // units in flight
#pragma unroll 1
    for (int j0 = 0; j0 < NU; j0 += kAhead) {
      float4 v[kAhead];
#pragma unroll
      for (int j = 0; j < kAhead; ++j)
        v[j] = own_unit(j0 + j, [&](int lr, int lc) { return __ldcg(Dt + lr * ld + lc); });
#pragma unroll
      for (int j = 0; j < kAhead; ++j)
        *reinterpret_cast<float4*>(snapR + unit_off(j0 + j, Col{})) = v[j];
    }
  }
  ++pc.d;
  pc.chunk += 2;
  stamp(3);
  return true;
}

// The parts of a FilterTask that follow from the tile (ti, tj) of round r.
template <typename T, int BS>
__device__ __forceinline__ FilterTask<T> filter_task(const Args<T>& a, int r, int ti, int tj) {
  const int64_t row0 = (int64_t)ti * BS, col0 = (int64_t)tj * BS, k0 = (int64_t)r * BS;
  FilterTask<T> f;
  f.D = a.D + row0 * a.ld + col0;
  f.P = a.P ? a.P + row0 * a.ld + col0 : nullptr;
  f.ld = a.ld;
  f.nrow = (int)(a.n - row0 < BS ? a.n - row0 : BS);
  f.ncol = (int)(a.n - col0 < BS ? a.n - col0 : BS);
  f.kn = (int)(a.n - k0 < BS ? a.n - k0 : BS);
  f.diag = ti == tj;
  f.status = a.status;
  f.q = q_scale(__ldcg(a.qexp + r));
  f.Psrc = nullptr;
  f.neg = false;
  return f;
}

// A remaining-tile task's FilterTask; its operands' bounds are in the ring stage st.
template <typename T, int BS, int LBS>
__device__ __forceinline__ FilterTask<T> tile_filter(const Args<T>& a, const fwh::Task& k,
                                                     unsigned char* smem, unsigned st) {
  using L = WsLayout<LBS, T>;
  FilterTask<T> f = filter_task<T, BS>(a, k.r, k.ti, k.tj);
  const size_t ta = (size_t)(k.r & 1) * a.slot_tiles + k.ti, tb = (size_t)(k.r & 1) * a.slot_tiles + k.tj;
  f.A = a.colR + ta * BS * BS;
  f.B = a.rowR + tb * BS * BS;
  f.old = reinterpret_cast<const T*>(smem + L::d_off());
  f.Ah = reinterpret_cast<const uint32_t*>(smem + L::ring_off() + st * L::kStage);
  f.Bh = f.Ah + KeysH<BS>::kTileWords;
  f.Psrc = a.rowP + tb * BS * BS;
  f.neg = __ldcg(a.colB + ta) | __ldcg(a.rowB + tb);
  return f;
}

// Releases the buffers of a remaining-tile task.  Whole warp.
__device__ __forceinline__ void leave_tile_f(WsBars* wb, PipeCnt& pc) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    mbar_arrive(&wb->chunk_empty[pc.chunk & 1]);
    mbar_arrive(&wb->d_empty);
  }
  ++pc.chunk;
  ++pc.d;
}

// Remaining-tile task of fp64 (BS = 64) over every step of every entry, after the
// filter's turn (ws_minplus_f) or, with kSkip, without it: the whole task.  Out of
// line and not called from ws_minplus_f, whose tiles paid 3 to 5 % for the call.
template <typename T, int BS, int LBS, bool kSkip>
__device__ __noinline__ bool ws_exact_f(const Args<T>& a, const fwh::Task& k, unsigned char* smem,
                                        WsBars* wb, PipeCnt& pc, uint64_t* tr) {
  const unsigned st = pc.chunk & 1;
  const long long t_a = tr ? clock64() : 0;
  if (kSkip) {
    const int group = (int)threadIdx.x >> 7;
    if (!mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, a.status, a.abort_flag, a.timeout_ns))
      return false;
    const long long cw = tr ? clock64() - t_a : 0;
    turn_wait(group);
    turn_pass(group ^ 1);
    const long long t_b = tr ? clock64() : 0;
    if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns)) return false;
    if (tr) {
      tr[7] = cyc20(clock64() - t_b) | (cyc20(cw) << 20);
      tr[8] = 0;
    }
  }
  int tx, ty;
  h_thread(tx, ty);
  relax_exact<T, BS, true>(tile_filter<T, BS, LBS>(a, k, smem, st), tx, ty);
  leave_tile_f(wb, pc);
  if (tr) {  // (the cycles of the relaxation come on top of the filter's)
    const uint64_t t = (uint64_t)(clock64() - t_a);
    tr[8] += t | t << 32;
  }
  return true;
}

// Remaining-tile task of fp64 (BS = 64): the 16-bit pass in turns, then the exact
// relaxation of the entries that may improve while the other group of warps has
// its turn.  The first rounds are bound by those relaxations, the later ones by the
// 16-bit pass (20 K SM cycles per tile, exact 160 K): n = 4096 133 -> 25.4 ms.
template <typename T, int BS, int LBS>
__device__ __noinline__ bool ws_minplus_f(const Args<T>& a, const fwh::Task& k, unsigned char* smem,
                                          WsBars* wb, PipeCnt& pc, uint64_t* tr, bool& exact) {
  using H = KeysH<BS>;
  using L = WsLayout<LBS, T>;
  constexpr int TM = Geo<BS>::TM;
  int tx, ty;
  h_thread(tx, ty);
  const unsigned st = pc.chunk & 1;
  const long long t_a = tr ? clock64() : 0;
  if (!mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, a.status, a.abort_flag, a.timeout_ns))
    return false;
  const long long cw = tr ? clock64() - t_a : 0;
  uint32_t acc[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) acc[m][nn] = 0xffffffffu;
  const int group = (int)threadIdx.x >> 7;
  turn_wait(group);
  const uint32_t* const As = reinterpret_cast<const uint32_t*>(smem + L::ring_off() + st * L::kStage);
  core_h<BS>(As, As + H::kTileWords, acc, tx, ty);
  turn_pass(group ^ 1);
  const long long t_b = tr ? clock64() : 0;
  if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns)) return false;
  if (tr) {
    tr[7] = cyc20(clock64() - t_b) | (cyc20(cw) << 20);
    tr[8] = (uint64_t)(t_b - t_a);
  }
  const FilterTask<T> f = tile_filter<T, BS, LBS>(a, k, smem, st);
  exact = !refine_tile<T, BS, true>(f, acc, tx, ty,
                                    reinterpret_cast<uint32_t*>(smem + L::scr_off() +
                                                                (threadIdx.x >> 5) * L::kScrWarp));
  if (!exact) leave_tile_f(wb, pc);
  if (tr) tr[8] |= (uint64_t)(clock64() - t_a) << 32;
  return true;
}

// 16-bit bounds of a BS x BS tile in shared memory (rows and columns at or
// beyond nrow, ncol: INF) as an A operand (steps along the columns) or a B
// operand (steps along the rows).  Returns 1 if an entry is negative.
template <typename T, int BS, bool kA, class Src>
__device__ __forceinline__ int quantize_tile(uint32_t* H, const QScale& q, Src&& src) {
  using Gm = Geo<BS>;
  constexpr int G = Gm::G, NW = KeysH<BS>::kNW;
  static_assert(NW == 2, "blocks of 64");
  int neg = 0;
#pragma unroll 1
  for (int i = threadIdx.x; i < BS * 16; i += kThreads) {
    const int x = kA ? i / 16 : i % BS, tk = kA ? i % 16 : i / BS;
    T v[2 * NW];
#pragma unroll
    for (int j = 0; j < 2 * NW; ++j) {
      const int kk = Gm::idx(tk, j);
      v[j] = src(kA ? x : kk, kA ? kk : x);
    }
    uint32_t word[NW];
#pragma unroll
    for (int e = 0; e < NW; ++e)
      word[e] = Quant<T>::q_of(v[e], q) | Quant<T>::q_of(v[e + NW], q) << 16;
#pragma unroll
    for (int j = 0; j < 2 * NW; ++j) neg |= v[j] < T(0) ? 1 : 0;
    const int t16 = (x % Gm::SPAN) / G, m = (x / Gm::SPAN) * G + x % G;  // x = idx(t16, m)
    uint32_t* u = H + h_unit<BS>(tk * NW / 4, m, t16) + tk * NW % 4;
    *reinterpret_cast<uint2*>(u) = make_uint2(word[0], word[1]);
  }
  return neg;
}

// (out of line, as ws_exact_f)
template <typename T, int BS>
__device__ __noinline__ void panel_exact(const FilterTask<T>& f, int tx, int ty) {
  relax_exact<T, BS, false>(f, tx, ty);
  __syncwarp();
}

// Panel task of round r of fp64 (BS = 64): Dbuf holds the tile's own values,
// ring stage s0 the closed pivot, and stage s1 takes the 16-bit bounds of
// both.  Filtered like a remaining tile, with its exact operands in shared
// memory; then the tile's snapshots (values, 16-bit bounds, a row tile's
// predecessors) are made from the relaxed tile.  A row tile's predecessors
// come from its own old ones, which wait in the snapshot's place meanwhile.
template <typename T, int BS, int LBS, bool is_row>
__device__ __noinline__ bool ws_panel_f(const Args<T>& a, const fwh::Task& k, unsigned char* smem,
                                        WsBars* wb, CtaScratch* cs, PipeCnt& pc) {
  using H = KeysH<BS>;
  using L = WsLayout<LBS, T>;
  constexpr int TM = Geo<BS>::TM;
  const int lane = threadIdx.x & 31;
  int tx, ty;
  h_thread(tx, ty);
  const int r = k.r, t = is_row ? k.tj : k.ti;
  const unsigned s0 = pc.chunk & 1, s1 = s0 ^ 1;
  const T* const own = reinterpret_cast<const T*>(smem + L::d_off());
  const T* const piv = reinterpret_cast<const T*>(smem + L::ring_off() + s0 * L::kStage);
  uint32_t* const Ah = reinterpret_cast<uint32_t*>(smem + L::ring_off() + s1 * L::kStage);
  uint32_t* const Bh = Ah + H::kTileWords;
  stamp(0);
  FilterTask<T> f = filter_task<T, BS>(a, r, k.ti, k.tj);
  const size_t tile = (size_t)(r & 1) * a.slot_tiles + t;
  int32_t* const snapP = a.rowP + tile * BS * BS;
  if (is_row && f.P) stage_tile_i32<BS>(snapP, a.P, a.n, a.ld, k.ti, k.tj, nullptr);
  if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns) ||
      !mbar_wait(&wb->chunk_full[s0], (pc.chunk >> 1) & 1, a.status, a.abort_flag,
                 a.timeout_ns) ||
      !mbar_wait(&wb->chunk_full[s1], ((pc.chunk + 1) >> 1) & 1, a.status, a.abort_flag,
                 a.timeout_ns))
    return false;
  auto own_at = [&](int i, int j) { return i < f.nrow && j < f.ncol ? own[i * BS + j] : Num<T>::inf(); };
  auto piv_at = [&](int i, int j) { return piv[i * BS + j]; };
  int neg[1];
  if constexpr (is_row)
    neg[0] = quantize_tile<T, BS, true>(Ah, f.q, piv_at) | quantize_tile<T, BS, false>(Bh, f.q, own_at);
  else
    neg[0] = quantize_tile<T, BS, true>(Ah, f.q, own_at) | quantize_tile<T, BS, false>(Bh, f.q, piv_at);
  block_max(neg, cs);
  bar_compute();  // (and the old predecessors are in place)
  stamp(1);
  uint32_t acc[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) acc[m][nn] = 0xffffffffu;
  core_h<BS>(Ah, Bh, acc, tx, ty);
  f.A = is_row ? piv : own;
  f.B = is_row ? own : piv;
  f.old = own;
  f.Ah = Ah;
  f.Bh = Bh;
  f.Psrc = is_row ? snapP : a.pivP + (size_t)(r & 1) * BS * BS;
  f.neg = neg[0] != 0;
  if (!refine_tile<T, BS, false>(f, acc, tx, ty,
                                 reinterpret_cast<uint32_t*>(smem + L::scr_off() +
                                                             (threadIdx.x >> 5) * L::kScrWarp)))
    panel_exact<T, BS>(f, tx, ty);
  fence_proxy_async_shared();  // generic writes before the stage's next TMA fill
  bar_compute();  // the relaxed tile is in the matrix, the operands are free
  stamp(2);
  if (lane == 0) {
    mbar_arrive(&wb->d_empty);
    mbar_arrive(&wb->chunk_empty[0]);
    mbar_arrive(&wb->chunk_empty[1]);
  }
  ++pc.d;
  pc.chunk += 2;
  T* const snapR = (is_row ? a.rowR : a.colR) + tile * BS * BS;
  uint32_t* const snapH = (is_row ? a.rowH : a.colH) + tile * H::kTileWords;
  if (is_row && f.P) stage_tile_i32<BS>(snapP, a.P, a.n, a.ld, k.ti, k.tj, nullptr);
  auto relaxed = [&](int i, int j) {
    const bool in = i < f.nrow && j < f.ncol;
    const T v = in ? __ldcg(f.D + i * f.ld + j) : Num<T>::inf();
    snapR[i * BS + j] = v;
    return v;
  };
  neg[0] = quantize_tile<T, BS, !is_row>(snapH, f.q, relaxed);
  block_max(neg, cs);
  if (threadIdx.x == 0) (is_row ? a.rowB : a.colB)[tile] = neg[0];
  stamp(3);
  return true;
}

// Remaining-tile task (phase 4 of round r, tile ti,tj) over packed 32-bit keys
// (kKeys; 16-bit keys: ws_minplus_h) or with compare and select.  kExpand: the
// operands may need to be expanded first (dec).  Keys that need not be have a loop
// of their own, in the kernel itself: a call in it, or out of line, its registers
// are laid out for the callee (int32 with weights to 3e5, n = 3000: 2.74 ms, one
// loop for both 2.78, out of line 2.85).  Returns false if an operand never
// arrived (the kernel then stops).
template <typename T, int BS, int LBS, bool kKeys, bool kExpand>
__device__ __forceinline__ bool ws_minplus_body(TileCtx<T> c, int ti, int tj, int dec,
                                        unsigned char* smem, WsBars* wb, PipeCnt& pc,
                                        uint64_t* tr) {
  if (!kKeys && !c.P) return ws_minplus_dist<T, BS, LBS>(c, ti, tj, dec, smem, wb, pc, tr);
  using Gm = Geo<BS>;
  using K = Keys<BS>;
  using L = WsLayout<LBS, T>;
  using C = WsChunk<BS, T>;
  constexpr int TM = Gm::TM, G = Gm::G;
  constexpr bool kPacked = Num<T>::kPacked;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const T* Dbuf = reinterpret_cast<const T*>(smem + L::d_off());
  unsigned char* ring = smem + L::ring_off();
  const int64_t row0 = (int64_t)ti * BS, col0 = (int64_t)tj * BS;
  const int nrow = (int)(c.n - row0 < BS ? c.n - row0 : BS);  // valid rows / columns of the tile
  const int ncol = (int)(c.n - col0 < BS ? c.n - col0 : BS);
  const bool full = nrow == BS && ncol == BS;

  // optional per-phase SM-cycle counts (trace): Dbuf wait, operand-chunk waits;
  // start to end of the relaxation, whole task
  const long long t_a = tr ? clock64() : 0;
  long long cw = 0;
  // 1. the tile's current values (rows/columns beyond n read as INF)
  if (!mbar_wait(&wb->d_full, pc.d & 1, c.status, c.abort_flag, c.timeout_ns)) return false;
  const long long t_b = tr ? clock64() : 0;
  T old[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lc0 = g * Gm::SPAN + tx * G;
      T tmp[G];
      vload_s<G>(tmp, Dbuf + lr * BS + lc0);
#pragma unroll
      for (int e = 0; e < G; ++e)
        old[m][g * G + e] = (lr < nrow && lc0 + e < ncol) ? tmp[e] : Num<T>::inf();
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(&wb->d_empty);
  ++pc.d;

  T* Drow = c.D + row0 * c.ld + col0;
  int32_t* Prow = c.P + row0 * c.ld + col0;
  bool neg = false;
  if constexpr (kKeys) {  // (packed keys: int32 only)
    uint32_t acc[TM][TM];
    int32_t omax = 0;
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) {
        acc[m][nn] = kPacked ? key_of<BS>((int32_t)old[m][nn]) : 0u;
        omax = max(omax, (int32_t)old[m][nn]);
      }
    const bool clamped = omax >= K::CAP;  // some old value's key is the clamp
    for (int ch = 0; ch < C::NC; ++ch) {
      const unsigned st = pc.chunk & 1;
      const long long w0 = tr ? clock64() : 0;
      if (!mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, c.status, c.abort_flag,
                     c.timeout_ns))
        return false;
      if (tr) cw += clock64() - w0;
      if constexpr (kExpand)
        decode_chunk<T, BS, C::CK>(ring + st * L::kStage, dec, ch, true);
      const uint32_t* As = reinterpret_cast<const uint32_t*>(ring + st * L::kStage);
      const uint32_t* Bs = As + C::CK * BS;
      core_packed<BS, C::CK>(As, Bs, acc, tx, ty);
      __syncwarp();
      if (lane == 0) mbar_arrive(&wb->chunk_empty[st]);
      ++pc.chunk;
    }
    const long long t_c = tr ? clock64() : 0;
    if (tr) {
      tr[7] = cyc20(t_b - t_a) | (cyc20(cw) << 20);
      tr[8] = (uint64_t)(t_c - t_a);
    }
    // predecessors as "via k" codes: k = r*BS + code - 1
    const int32_t via0 = via_code((int64_t)c.r * BS - 1);  // via_code(k) = via0 - code
    // most tasks of later rounds improve nothing in a warp's 16 x 128 rows:
    // one OR over the codes and a vote skip the epilogue
    uint32_t any = 0;
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) any |= acc[m][nn];
    if (__any_sync(0xffffffffu, (any & K::MASK) != 0)) {
      if (full && !__any_sync(0xffffffffu, clamped)) {
        // no clamped key in the warp: every key decodes exactly; a group of
        // G entries with an improvement is stored as one 16-byte vector
#pragma unroll
        for (int m = 0; m < TM; ++m) {
          const int lr = Gm::idx(ty, m);
#pragma unroll
          for (int g = 0; g < Gm::NG; ++g) {
            const int lc0 = g * Gm::SPAN + tx * G;
            uint32_t cg = 0;
            T dv[G];
#pragma unroll
            for (int e = 0; e < G; ++e) {
              const uint32_t kv = acc[m][g * G + e];
              cg |= kv & K::MASK;
              dv[e] = (T)(int32_t)(kv >> K::KB);
            }
            if (cg) vstore<G>(Drow + lr * c.ld + lc0, dv);
            if (c.P) {
#pragma unroll
              for (int e = 0; e < G; ++e) {
                const int code = (int)(acc[m][g * G + e] & K::MASK);
                if (code) Prow[lr * c.ld + lc0 + e] = via0 - code;
              }
            }
          }
        }
      } else {
        // improved entries one by one (a clamped key -- old value CAP or
        // more, INF or a large finite one -- keeps its old value)
#pragma unroll
        for (int m = 0; m < TM; ++m) {
          const int lr = Gm::idx(ty, m);
#pragma unroll
          for (int nn = 0; nn < TM; ++nn) {
            const int code = (int)(acc[m][nn] & K::MASK);
            const int lc = Gm::idx(tx, nn);
            if (code && lr < nrow && lc < ncol) {
              Drow[lr * c.ld + lc] = (T)(int32_t)(acc[m][nn] >> K::KB);
              if (c.P) Prow[lr * c.ld + lc] = via0 - code;
            }
          }
        }
      }
    }
  } else {
    constexpr bool kHold = kPredSmem<T, BS>;  // the stage stays: its predecessors are read below
    static_assert(!kHold || C::NC == 1, "all of a tile's operands in one stage");
    const unsigned st0 = pc.chunk & 1;
    int arg[TM][TM];
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) arg[m][nn] = 0;
    for (int ch = 0; ch < C::NC; ++ch) {
      const unsigned st = pc.chunk & 1;
      const long long w0 = tr ? clock64() : 0;
      if (!mbar_wait(&wb->chunk_full[st], (pc.chunk >> 1) & 1, c.status, c.abort_flag,
                     c.timeout_ns))
        return false;
      if (tr) cw += clock64() - w0;
      decode_chunk<T, BS, C::CK>(ring + st * L::kStage, dec, ch, false);
      const T* As = reinterpret_cast<const T*>(ring + st * L::kStage);
      const T* Bs = As + C::CK * BS;
      core_generic<BS, T, C::CK, false>(As, Bs, old, arg, tx, ty, ch * C::CK);
      __syncwarp();
      if (!kHold && lane == 0) mbar_arrive(&wb->chunk_empty[st]);
      ++pc.chunk;
    }
    argmin_finish<T>(arg);
    const long long t_c = tr ? clock64() : 0;
    if (tr) {
      tr[7] = cyc20(t_b - t_a) | (cyc20(cw) << 20);
      tr[8] = (uint64_t)(t_c - t_a);
    }
    const int32_t via0 = via_code((int64_t)c.r * BS - 1);
    const int32_t* const Psrc =
        reinterpret_cast<const int32_t*>(ring + st0 * L::kStage + 2 * C::kChunkBytes);
#pragma unroll
    for (int m = 0; m < TM; ++m) {
      const int lr = Gm::idx(ty, m);
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) {
        const int lc = Gm::idx(tx, nn);
        if (arg[m][nn] && lr < nrow && lc < ncol) {
          Drow[lr * c.ld + lc] = old[m][nn];
          Prow[lr * c.ld + lc] =
              kHold ? Psrc[(arg[m][nn] - 1) * BS + lc] : via0 - arg[m][nn];
          neg |= (row0 + lr == col0 + lc) && old[m][nn] < T(0);
        }
      }
    }
    if (kHold) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&wb->chunk_empty[st0]);
    }
  }
  if (tr) tr[8] |= (uint64_t)(clock64() - t_a) << 32;  // whole task
  if (neg) atomicOr(c.status, kStNegCycle);
  return true;
}

// Out of line: every other case.
template <typename T, int BS, int LBS, bool kKeys, bool kExpand>
__device__ __noinline__ bool ws_minplus(TileCtx<T> c, int ti, int tj, int dec,
                                        unsigned char* smem, WsBars* wb, PipeCnt& pc,
                                        uint64_t* tr) {
  return ws_minplus_body<T, BS, LBS, kKeys, kExpand>(c, ti, tj, dec, smem, wb, pc, tr);
}

// Relaxation and epilogue of a producer-fed panel task (ws_panel) whose
// operands are staged: packed keys (kFast) or raw values, A transposed in the
// scratch stage, B in natural layout (Dbuf for a row tile, the pivot stage
// for a column tile).  The accumulators start from the tile's own values as
// staged there.  A function of its own per path, so that the two register
// sets are never live together.
template <typename T, int BS, int LBS, bool is_row, bool kFast>
__device__ __noinline__ bool ws_panel_finish(const Args<T>& a, int r, int t, T* Dbuf, T* Piv,
                                             unsigned char* scratch, WsBars* wb, CtaScratch* cs,
                                             PipeCnt& pc) {
  using Gm = Geo<BS>;
  using K = Keys<BS>;
  constexpr int TM = Gm::TM, G = Gm::G;
  using U = std::conditional_t<kFast, uint32_t, T>;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const U* As = reinterpret_cast<const U*>(scratch);
  const U* Bs = reinterpret_cast<const U*>(is_row ? Dbuf : Piv);
  U acc[TM][TM];
  if constexpr (is_row) {
    // own values: B-form in Dbuf
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int g = 0; g < Gm::NG; ++g) {
        U v[G];
        vload_s<G>(v, Bs + Gm::idx(ty, m) * BS + g * Gm::SPAN + tx * G);
#pragma unroll
        for (int e = 0; e < G; ++e) acc[m][g * G + e] = v[e];
      }
  } else {
    // own values: A-form in the scratch stage (keys with their column's code)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn)
#pragma unroll
      for (int g = 0; g < Gm::NG; ++g) {
        U v[G];
        vload_s<G>(v, As + Gm::idx(tx, nn) * BS + g * Gm::SPAN + ty * G);
#pragma unroll
        for (int e = 0; e < G; ++e) {
          if constexpr (kFast) acc[g * G + e][nn] = v[e] & ~K::MASK;
          else acc[g * G + e][nn] = v[e];
        }
      }
  }
  int code[kFast ? 1 : TM][kFast ? 1 : TM];
  if constexpr (kFast) {
    core_packed<BS>(As, Bs, acc, tx, ty);
  } else {
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) code[m][nn] = 0;
    core_generic<BS, T>(As, Bs, acc, code, tx, ty);
  }
  // operands consumed: order this warp's shared-memory writes before the
  // copies that will overwrite the buffers, then release them
  fence_proxy_async_shared();
  __syncwarp();
  if (lane == 0) {
    const unsigned s0 = pc.chunk & 1;
    mbar_arrive(&wb->d_empty);
    mbar_arrive(&wb->chunk_empty[s0]);
    mbar_arrive(&wb->chunk_empty[s0 ^ 1]);
  }
  ++pc.d;
  pc.chunk += 2;
  stamp(2);

  // new values: their bound (the remaining tiles' packed-key test)
  auto value = [&](int m, int nn) -> T {
    if constexpr (kFast) {
      const int32_t v = (int32_t)(acc[m][nn] >> K::KB);
      return v == K::CAP ? Num<T>::inf() : (T)v;
    } else {
      return acc[m][nn];
    }
  };
  auto codeof = [&](int m, int nn) -> int {
    if constexpr (kFast) return (int)(acc[m][nn] & K::MASK);
    else return code[m][nn];
  };
  // (fast path: the accumulator without its code is the value's key)
  auto key = [&](int m, int nn) -> uint32_t {
    if constexpr (kFast) return acc[m][nn] & ~K::MASK;
    else return key_of<BS>((int32_t)acc[m][nn]);
  };
  int nb, has_inf;
  if constexpr (kFast) {
    // (as Bound32, on the keys: values from CAP are INF, none is negative)
    constexpr uint32_t kTop = 0u - ((uint32_t)K::CAP << K::KB);
    uint32_t top = 0, hi = 0;
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) {
        top = __viaddmax_u32(acc[m][nn], kTop, top);
        hi = max(hi, acc[m][nn]);
      }
    nb = top >= kTop ? (int)((top - kTop) >> K::KB) : 0;
    has_inf = (int)(hi >> K::KB) >= K::CAP ? kBndInf : 0;
  } else {
    Bound32<BS> b;
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) b.add((int32_t)acc[m][nn]);
    nb = b.bound();
    has_inf = b.inf();
  }
  block_max2(nb, has_inf, cs);
  // snapshots: 32-bit keys, which are exact while every finite value is below CAP;
  // beyond that the raw values as well, and without packed keys the raw values
  // only.  16-bit keys too where the bound allows them (16-bit keys alone, expanded
  // where the other operand of a tile has none: a grid of n = 8100 34.2 ms, 31.8
  // with both; n = 8000 of degree 8, weights to 100, 35.1 and 34.5).
  const bool hok = a.packed && h_tile_ok<BS>(nb | has_inf);
  const bool keys = a.packed != 0;
  const bool raw = !a.packed || nb >= K::CAP;
  const int slot = r & 1;
  const size_t tile_off = ((size_t)slot * a.slot_tiles + t) * BS * BS;
  // the pointers and sizes in registers: through the reference every access
  // would be a load, repeated after each store (which might alias it)
  T* const D = a.D;
  int32_t* const P = a.P;
  const int64_t n = a.n, ld = a.ld;
  uint32_t* const snapK = (is_row ? a.rowK : a.colK) + tile_off;
  T* const snapR = (is_row ? a.rowR : a.colR) + tile_off;
  int32_t* const bnd = (is_row ? a.rowB : a.colB) + (size_t)slot * a.slot_tiles + t;

  // the live tile (values, and via codes k = r*BS + code - 1 where improved);
  // a row tile's snapshots in the same (B-form) order
  const int32_t via0 = via_code((int64_t)r * BS - 1);
  const int ti = is_row ? r : t, tj = is_row ? t : r;
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
    const int64_t gi = (int64_t)ti * BS + lr;
#pragma unroll
    for (int gg = 0; gg < Gm::NG; ++gg) {
      const int lc0 = gg * Gm::SPAN + tx * G;
      const int64_t gj0 = (int64_t)tj * BS + lc0;
      T vs[G];
      int32_t vp[G];
      bool all = true;
      int cq[G];
#pragma unroll
      for (int q = 0; q < G; ++q) {
        vs[q] = value(m, gg * G + q);
        cq[q] = codeof(m, gg * G + q);
        vp[q] = via0 - cq[q];
        all &= cq[q] != 0;
      }
      if (gi < n) {
        if (gj0 + G <= n) {
          vstore<G>(D + gi * ld + gj0, vs);
          if (P) {
            if (all) {
              vstore<G>(P + gi * ld + gj0, vp);  // (early rounds: most groups)
            } else {
#pragma unroll
              for (int q = 0; q < G; ++q)
                if (cq[q]) P[gi * ld + gj0 + q] = vp[q];
            }
          }
        } else {
#pragma unroll
          for (int q = 0; q < G; ++q)
            if (gj0 + q < n) {
              D[gi * ld + gj0 + q] = vs[q];
              if (P && cq[q]) P[gi * ld + gj0 + q] = vp[q];
            }
        }
      }
      if constexpr (is_row) {
        if (keys) {
          uint32_t kq[G];
#pragma unroll
          for (int q = 0; q < G; ++q) kq[q] = key(m, gg * G + q);
          vstore<G>(snapK + lr * BS + lc0, kq);
        }
        if (raw) vstore<G>(snapR + lr * BS + lc0, vs);
      }
    }
  }
  if constexpr (!is_row) {
    // a column tile's snapshots: A-form (transposed), keys with code = column + 1
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) {
      const int lc = Gm::idx(tx, nn);
#pragma unroll
      for (int g = 0; g < Gm::NG; ++g) {
        const size_t off = (size_t)lc * BS + g * Gm::SPAN + ty * G;
        if (keys) {
          uint32_t kq[G];
#pragma unroll
          for (int e = 0; e < G; ++e) kq[e] = key(g * G + e, nn) + (uint32_t)lc + 1u;
          vstore<G>(snapK + off, kq);
        }
        if (raw) {
          T vs[G];
#pragma unroll
          for (int e = 0; e < G; ++e) vs[e] = value(g * G + e, nn);
          vstore<G>(snapR + off, vs);
        }
      }
    }
  }
  if (hok) {
    // 16-bit keys: INF is the only value at or above the clamp
    uint32_t* const snapH = (is_row ? a.rowH : a.colH) +
                            ((size_t)slot * a.slot_tiles + t) * KeysH<BS>::kTileWords;
    auto key16 = [&](int m, int nn) -> uint32_t {
      const uint32_t v = (uint32_t)min((int32_t)value(m, nn), KeysH<BS>::kCapF);
      return (has_inf ? min(v, (uint32_t)KeysH<BS>::kCapI) : v) << KeysH<BS>::KB;
    };
    if constexpr (is_row)
      put_h<BS, false>(snapH, ty, tx, [&](int k, int q) { return key16(k, q); });
    else
      put_h<BS, true>(snapH, tx, ty, [&](int k, int q) { return key16(q, k); });
  }
  if (tid == 0) *bnd = nb | has_inf | (hok ? kBndH : 0) | (keys ? kBndK : 0);
  stamp(3);
  return true;
}

// Relaxation over 16-bit keys and results of a producer-fed panel task whose
// operands are staged in the scratch stage (A at its start, then B); the
// tile's own values are in Dbuf, cap is the clamp of the operands' keys.  The
// live tile and the 16-bit snapshot are formed in the two ring stages and the
// publisher stores them in bulk (store_panel).  The accumulators go through
// shared memory and a short loop decodes them row by row: decoded in registers,
// with a branch and a scattered store for each of 64 entries, they took 8-14 K SM
// cycles, the loop 3 K.  The results'
// finite values are below cap, so the tile always has a 16-bit snapshot and
// needs no other.
template <typename T, int BS, int LBS, bool is_row>
__device__ __forceinline__ void ws_panel_h(const Args<T>& a, int r, int t, int cap,
                                           unsigned char* smem, WsBars* wb, CtaScratch* cs,
                                           PipeCnt& pc, unsigned pslot) {
  using Gm = Geo<BS>;
  using H = KeysH<BS>;
  using L = WsLayout<LBS, T>;
  constexpr int TM = Gm::TM, G = Gm::G, NW = H::kNW;
  int tx, ty;
  h_thread(tx, ty);
  const unsigned s0 = pc.chunk & 1, s1 = s0 ^ 1;
  const T* const own = reinterpret_cast<const T*>(smem + L::d_off());
  uint32_t* const tile = reinterpret_cast<uint32_t*>(smem + L::ring_off() + s0 * L::kStage);
  uint32_t* const hst = reinterpret_cast<uint32_t*>(smem + L::ring_off() + s1 * L::kStage);
  uint32_t acc[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) acc[m][nn] = 0xffffffffu;
  core_h<BS>(hst, hst + H::kTileWords, acc, tx, ty);
  stamp(2);
  put_tile<BS, false>(tile, acc, tx, ty);  // (the pivot it held is in the operands)
  bar_compute();                           // every warp has left the operands

  const int64_t row0 = (int64_t)(is_row ? r : t) * BS, col0 = (int64_t)(is_row ? t : r) * BS;
  const int64_t n = a.n, ld = a.ld;
  const int nrow = (int)(n - row0 < BS ? n - row0 : BS);
  const int ncol = (int)(n - col0 < BS ? n - col0 : BS);
  const bool whole = nrow == BS && ncol == BS;
  T* const D = a.D + row0 * ld + col0;
  int32_t* const P = a.P ? a.P + row0 * ld + col0 : nullptr;
  const int32_t via0 = via_code((int64_t)r * BS);  // via_code(k) = via0 - kk
  int res[2] = {0, 0};  // bound of the finite results; any INF
  // the 16-bit snapshot words of thread row tk along the inner dimension and
  // operand row x, and the tile's entries behind them
#pragma unroll 1
  for (int i = threadIdx.x; i < BS * 16; i += kThreads) {
    const int x = is_row ? i % BS : i / 16, tk = is_row ? i / BS : i % 16;
    uint32_t word[NW], sum[2 * NW];
    T v[2 * NW];
    auto at = [&](int j) {  // entry j: half j / NW of word j % NW
      const int kk = Gm::idx(tk, j);
      return (is_row ? kk : x) * BS + (is_row ? x : kk);
    };
#pragma unroll
    for (int j = 0; j < 2 * NW; ++j) {
      sum[j] = tile[at(j)];
      v[j] = own[at(j)];
    }
#pragma unroll
    for (int e = 0; e < NW; ++e)
      word[e] = is_row ? 0u : (uint32_t)Gm::idx(tk, e) | ((uint32_t)Gm::idx(tk, e + NW) << 16);
#pragma unroll
    for (int j = 0; j < 2 * NW; ++j) {
      const uint32_t mm = min(sum[j] & 0xffffu, sum[j] >> 16);
      const int d = (int)(mm >> H::KB);
      const int lr = at(j) / BS, lc = at(j) % BS;
      const bool in = lr < nrow && lc < ncol;
      const bool better = in && d < (int)v[j] && d < cap;
      v[j] = better ? (T)d : in ? v[j] : Num<T>::inf();
      const bool inf = !Num<T>::finite(v[j]);
      tile[at(j)] = (uint32_t)v[j];
      word[j % NW] += (uint32_t)(inf ? H::kCapI : (int)v[j]) << (H::KB + 16 * (j / NW));
      res[0] = max(res[0], inf ? 0 : (int)v[j]);
      res[1] |= inf ? 1 : 0;
      if (P && better) P[lr * ld + lc] = via0 - (int32_t)(mm & H::MASK);
    }
    if (!whole) {
#pragma unroll 1
      for (int j = 0; j < 2 * NW; ++j) {
        const int lr = at(j) / BS, lc = at(j) % BS;
        if (lr < nrow && lc < ncol) D[lr * ld + lc] = (T)tile[lr * BS + lc];
      }
    }
    const int t16 = (x % Gm::SPAN) / G, m = (x / Gm::SPAN) * G + x % G;  // x = idx(t16, m)
    uint32_t* u = hst + h_unit<BS>(tk * NW / 4, m, t16) + tk * NW % 4;
    if constexpr (NW == 4) *reinterpret_cast<uint4*>(u) = make_uint4(word[0], word[1], word[2], word[3]);
    else if constexpr (NW == 2) *reinterpret_cast<uint2*>(u) = make_uint2(word[0], word[1]);
    else *u = word[0];
  }
  // (the publisher releases the ring stages)
  fence_proxy_async_shared();
  pc.chunk += 2;
  block_max(res, cs);
  if ((threadIdx.x & 31) == 0) mbar_arrive(&wb->d_empty);
  ++pc.d;
  if (threadIdx.x == 0) {
    ((is_row ? a.rowB : a.colB) + (size_t)(r & 1) * a.slot_tiles)[t] =
        res[0] | (res[1] ? kBndInf : 0) | kBndH;
    wb->pst[pslot] = kPstOn | (s0 ? kPstStage : 0) | (whole ? kPstTile : 0);
  }
  stamp(3);
}

// Publisher's part of a 16-bit panel task: the bulk stores of its results from
// shared memory, the release of the ring stages once they have been read, and
// the wait for the stores themselves (the publication follows).  Whole warp.
template <typename T, int BS, int LBS>
__device__ void store_panel(const Args<T>& a, const fwh::Task& k, int pst, unsigned char* smem,
                            WsBars* wb, int lane) {
  using L = WsLayout<LBS, T>;
  const bool is_row = k.type == 1;
  const unsigned s0 = (pst & kPstStage) ? 1 : 0, s1 = s0 ^ 1;
  const size_t ht = (size_t)(k.r & 1) * a.slot_tiles + (is_row ? k.tj : k.ti);
  const int64_t row0 = (int64_t)k.ti * BS, col0 = (int64_t)k.tj * BS;
  const T* const tile = reinterpret_cast<const T*>(smem + L::ring_off() + s0 * L::kStage);
  if (lane == 0) {
    bulk_s2g((is_row ? a.rowH : a.colH) + ht * KeysH<BS>::kTileWords,
             smem + L::ring_off() + s1 * L::kStage, (unsigned)(BS * BS * 2));
    if ((pst & kPstTile) && a.tmapD) tma_store_2d(a.tmapD, (int)col0, (int)row0, tile);
  }
  if ((pst & kPstTile) && !a.tmapD)
    for (int rr = lane; rr < BS; rr += 32)
      bulk_s2g(a.D + (row0 + rr) * a.ld + col0, tile + rr * BS, (unsigned)(BS * sizeof(T)));
  bulk_commit_wait_read();
  __syncwarp();
  if (lane == 0) {
    mbar_arrive_n(&wb->chunk_empty[0], kThreads / 32);
    mbar_arrive_n(&wb->chunk_empty[1], kThreads / 32);
  }
  bulk_wait_all();
  __syncwarp();
}

// Panel task of round r (int32), fed by the producer like a remaining tile:
// Dbuf holds the tile's own values, ring stage s0 the closed pivot (snapshot
// of slot r&1, natural layout) and stage s1 is scratch for the transposed A
// operand.  Row tile (r, t):    A = pivot (transposed), B = own old values.
// Column tile (t, r): A = own old values (transposed), B = pivot.
// The product with the closed pivot equals the in-place sequential phases 2
// and 3 (Sec. 2.3).  Predecessors are recorded as via codes (ViaPred), so the
// task needs no predecessor tile.  The operand buffers are released right
// after the relaxation: the producer streams the next task's operands while
// this one stores its results.
template <typename T, int BS, int LBS, bool is_row>
__device__ __noinline__ bool ws_panel(const Args<T>& a, const fwh::Task& k, unsigned char* smem,
                                      WsBars* wb, CtaScratch* cs, PipeCnt& pc, unsigned slot) {
  static_assert(Num<T>::kPacked, "producer-fed panels are the int32 path");
  using Gm = Geo<BS>;
  using K = Keys<BS>;
  using L = WsLayout<LBS, T>;
  static_assert(WsChunk<BS, T>::kTile <= L::kStage, "a tile per ring stage");
  constexpr int TM = Gm::TM, G = Gm::G;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if (threadIdx.x == 0) wb->pst[slot] = 0;
  const int r = k.r, t = is_row ? k.tj : k.ti;
  const int64_t row0 = (int64_t)k.ti * BS, col0 = (int64_t)k.tj * BS;
  const int nrow = (int)(a.n - row0 < BS ? a.n - row0 : BS);
  const int ncol = (int)(a.n - col0 < BS ? a.n - col0 : BS);
  T* Dbuf = reinterpret_cast<T*>(smem + L::d_off());
  const unsigned s0 = pc.chunk & 1, s1 = s0 ^ 1;
  T* Piv = reinterpret_cast<T*>(smem + L::ring_off() + s0 * L::kStage);
  unsigned char* scratch = smem + L::ring_off() + s1 * L::kStage;
  stamp(0);
  if (!mbar_wait(&wb->d_full, pc.d & 1, a.status, a.abort_flag, a.timeout_ns) ||
      !mbar_wait(&wb->chunk_full[s0], (pc.chunk >> 1) & 1, a.status, a.abort_flag,
                 a.timeout_ns) ||
      !mbar_wait(&wb->chunk_full[s1], ((pc.chunk + 1) >> 1) & 1, a.status, a.abort_flag,
                 a.timeout_ns))
    return false;

  // micro-tiles of the tile (entries beyond n read as INF) and of the pivot
  T s[TM][TM], pv[TM][TM];
#pragma unroll
  for (int m = 0; m < TM; ++m) {
    const int lr = Gm::idx(ty, m);
#pragma unroll
    for (int g = 0; g < Gm::NG; ++g) {
      const int lc0 = g * Gm::SPAN + tx * G;
      T ts[G], tp[G];
      vload_s<G>(ts, Dbuf + lr * BS + lc0);
      vload_s<G>(tp, Piv + lr * BS + lc0);
#pragma unroll
      for (int e = 0; e < G; ++e) {
        s[m][g * G + e] = (lr < nrow && lc0 + e < ncol) ? ts[e] : Num<T>::inf();
        pv[m][g * G + e] = tp[e];
      }
    }
  }
  // bounds of the tile and of the pivot, and whether they have an INF
  Bound32<BS> bown, bpiv;
#pragma unroll
  for (int m = 0; m < TM; ++m)
#pragma unroll
    for (int nn = 0; nn < TM; ++nn) {
      bown.add((int32_t)s[m][nn]);
      bpiv.add((int32_t)pv[m][nn]);
    }
  int bnd[4] = {bown.bound(), bpiv.bound(), bown.inf(), bpiv.inf()};
  block_max(bnd, cs);  // (its barriers also end every read of the raw buffers)
  const bool fast = a.packed && (bnd[0] + bnd[1] < K::CAP);
  if (a.packed) {
    if (const int cap = h_clamp<BS>(bnd[0] | bnd[2] | kBndH, bnd[1] | bnd[3] | kBndH)) {
      // 16-bit operands in the scratch stage: A, then B
      auto key16 = [&](T v) -> uint32_t { return (uint32_t)min((int)v, cap) << KeysH<BS>::KB; };
      uint32_t* const Ah = reinterpret_cast<uint32_t*>(scratch);
      uint32_t* const Bh = Ah + KeysH<BS>::kTileWords;
      if constexpr (is_row) {
        put_h<BS, true>(Ah, tx, ty, [&](int kr, int q) { return key16(pv[q][kr]); });
        put_h<BS, false>(Bh, ty, tx, [&](int kr, int q) { return key16(s[kr][q]); });
      } else {
        put_h<BS, true>(Ah, tx, ty, [&](int kr, int q) { return key16(s[q][kr]); });
        put_h<BS, false>(Bh, ty, tx, [&](int kr, int q) { return key16(pv[kr][q]); });
      }
      bar_compute();
      stamp(1);
      ws_panel_h<T, BS, LBS, is_row>(a, r, t, cap, smem, wb, cs, pc, slot);
      return true;
    }
  }

  // operands: A (transposed) into the scratch stage, B in place (natural
  // layout: the own tile in Dbuf for a row tile, the pivot for a column
  // tile).  Keys are formed in the registers of s and pv (int32), so that the
  // accumulators are only loaded once those are dead.
  uint32_t* Bk = reinterpret_cast<uint32_t*>(is_row ? (void*)Dbuf : (void*)Piv);
  if (fast) {
    uint32_t (&ka)[TM][TM] = reinterpret_cast<uint32_t(&)[TM][TM]>(is_row ? pv : s);
    uint32_t (&kb)[TM][TM] = reinterpret_cast<uint32_t(&)[TM][TM]>(is_row ? s : pv);
#pragma unroll
    for (int m = 0; m < TM; ++m)
#pragma unroll
      for (int nn = 0; nn < TM; ++nn) {
        const uint32_t cc = (uint32_t)Gm::idx(tx, nn) + 1u;  // the A entry's kk + 1
        ka[m][nn] = key_of<BS>((int32_t)ka[m][nn]) + cc;
        kb[m][nn] = key_of<BS>((int32_t)kb[m][nn]);
      }
    put_tile<BS, true>(reinterpret_cast<uint32_t*>(scratch), ka, tx, ty);
    put_tile<BS, false>(Bk, kb, tx, ty);
  } else {
    if constexpr (is_row) {
      put_tile<BS, true>(reinterpret_cast<T*>(scratch), pv, tx, ty);
      put_tile<BS, false>(Dbuf, s, tx, ty);  // (entries beyond n as INF)
    } else {
      put_tile<BS, true>(reinterpret_cast<T*>(scratch), s, tx, ty);
    }
  }
  bar_compute();
  stamp(1);
  return fast ? ws_panel_finish<T, BS, LBS, is_row, true>(a, r, t, Dbuf, Piv, scratch, wb, cs, pc)
              : ws_panel_finish<T, BS, LBS, is_row, false>(a, r, t, Dbuf, Piv, scratch, wb, cs,
                                                           pc);
}

// Any task, compute-warp side.
template <typename T, int BS, int LBS>
__device__ bool compute_task(const Args<T>& a, const fwh::Task& k, int mode, int dec,
                             unsigned char* smem, WsBars* wb, CtaScratch* cs, PipeCnt& pc,
                             unsigned slot, uint64_t* tr) {
  using L = WsLayout<LBS, T>;
  // pivot and panel tasks: SM cycles to operands staged | relaxed ; stored |
  // end (pivot: loads | steps ; predecessors resolved | end)
  auto trace_stamps = [&] {
    if (!tr) return;
    const long long t0 = t_stamp[0], t_end = clock64();
    tr[7] = (uint64_t)(t_stamp[1] - t0) | ((uint64_t)(t_stamp[2] - t0) << 32);
    tr[8] = (uint64_t)(t_stamp[3] - t0) | ((uint64_t)(t_end - t0) << 32);
  };
  if (k.type == 3 || k.type == kFusedTask) {
    bool ok;
    if constexpr (Num<T>::kPacked) {
      const TileCtx<T> ctx{a.D, a.P, a.n, a.ld, k.r, a.status, a.abort_flag, a.timeout_ns};
      if (mode > 1)
        ok = ws_minplus_h<T, BS, LBS>(a, k, mode, smem, wb, pc, tr);
      else if (mode && !(dec & (kFormHA | kFormHB)))
        ok = ws_minplus_body<T, BS, LBS, true, false>(ctx, k.ti, k.tj, 0, smem, wb, pc, tr);
      else if (mode)
        ok = ws_minplus<T, BS, LBS, true, true>(ctx, k.ti, k.tj, dec, smem, wb, pc, tr);
      else
        ok = ws_minplus<T, BS, LBS, false, true>(ctx, k.ti, k.tj, dec, smem, wb, pc, tr);
    } else if constexpr (sizeof(T) == 4) {
      ok = a.P ? ws_minplus_q<BS, LBS, true>(a, k, smem, wb, pc, tr)
               : ws_minplus_q<BS, LBS, false>(a, k, smem, wb, pc, tr);
    } else if constexpr (kFiltered<T, BS>) {
      if (skip_filter(pc.exact, k.r, k.ti, k.tj)) {
        ok = ws_exact_f<T, BS, LBS, true>(a, k, smem, wb, pc, tr);
      } else {
        bool exact = false;
        ok = ws_minplus_f<T, BS, LBS>(a, k, smem, wb, pc, tr, exact);
        if (exact) {
          pc.exact = k.r;
          ok = ws_exact_f<T, BS, LBS, false>(a, k, smem, wb, pc, tr);
        }
      }
    } else {
      const TileCtx<T> ctx{a.D, a.P, a.n, a.ld, k.r, a.status, a.abort_flag, a.timeout_ns};
      ok = ws_minplus_body<T, BS, LBS, false, false>(ctx, k.ti, k.tj, 0, smem, wb, pc, tr);
    }
    if (!ok || k.type == 3) return ok;
    // fused: the tile's stores precede the pivot's loads of it (same CTA),
    // and every warp has left the tile's operand buffers before the pivot
    // reuses them
    bar_compute();
    task_pivot<T, BS>(a, k.r + 1, smem + L::ring_off(), cs);
    bar_compute();
    return true;
  }
  if (k.type != 0 && !kOwnPanels<T, BS>) {
    bool ok = true;
    if constexpr (kOwnPanels<T, BS>) {
    } else if constexpr (Num<T>::kPacked)
      ok = k.type == 1 ? ws_panel<T, BS, LBS, true>(a, k, smem, wb, cs, pc, slot)
                       : ws_panel<T, BS, LBS, false>(a, k, smem, wb, cs, pc, slot);
    else if constexpr (sizeof(T) == 4)
      ok = k.type == 1 ? ws_panel_q<BS, LBS, true>(a, k, smem, wb, pc)
                       : ws_panel_q<BS, LBS, false>(a, k, smem, wb, pc);
    else
      ok = k.type == 1 ? ws_panel_f<T, BS, LBS, true>(a, k, smem, wb, cs, pc)
                       : ws_panel_f<T, BS, LBS, false>(a, k, smem, wb, cs, pc);
    if (ok) trace_stamps();
    return ok;
  }
  // Pivot tasks (and the exact 64-bit kernels' panels) overwrite the ring and
  // Dbuf from their first instructions: every compute warp must have left the
  // previous task (a slow warp may still be reading its last operands) before
  // any warp starts.
  bar_compute();
  if (k.type == 0)
    task_pivot<T, BS>(a, k.r, smem + L::ring_off(), cs);
  else if constexpr (kOwnPanels<T, BS>)
    task_panel<T, BS>(a, k.r, k.type == 1 ? k.tj : k.ti, k.type == 1, smem + L::ring_off(), cs);
  bar_compute();
  trace_stamps();
  return true;
}

// ----------------------------------------------------------- producer side ----

// Bounded wait until *p >= target (producer lane only).  Gives up when another
// CTA has aborted or when the wait exceeds timeout_ns; then records the
// timeout and raises the abort flag so that every CTA stops.
__device__ __forceinline__ bool wait_ge(const int* p, int target, int* abort_flag, int* status,
                                        int64_t timeout_ns) {
  if (ld_acquire(p) >= target) return true;
  const uint64_t t0 = globaltimer();
  // iteration cap as well as the clock: each iteration sleeps >= 32 ns
  const int64_t max_it = timeout_ns / 32 + 1024;
  // sleeps back off to 64 ns at most: a flag is polled soon after it is
  // published (n = 1024 at BS = 32: 0.610 -> 0.606 ms against 256 ns; the
  // large solves and the batched workload unchanged)
  unsigned ns = 32;
  for (int64_t it = 0;; ++it) {
    __nanosleep(ns);
    if (ns < 64) ns <<= 1;
    if (ld_acquire(p) >= target) return true;
    if (ld_relaxed(abort_flag)) return false;
    if (globaltimer() - t0 > (uint64_t)timeout_ns || it > max_it) {
      atomicOr(status, kStTimeout);
      atomicExch(abort_flag, 1);
      return false;
    }
  }
}

// Inputs of task k (Sec. 2.3 blocked-FW phase order, Opt-9's per-block dependencies of
// Sec. 3.2, and the slot reuse of the double-buffered snapshots): dependency
// `lane` (0..2) as a counter and the value it must reach; false when the task
// has fewer.
template <typename T>
__device__ __forceinline__ bool dep_of(const Args<T>& a, const fwh::Task& k, int lane,
                                       const int*& p, int& target) {
  const int R = a.R;
  const int* ver = a.ver;
  // Slot reuse is guarded by per-round counts: tasks of different rounds may
  // finish out of order, so a running total could reach its target while a
  // task of round r-2 still reads the slot.
  switch (k.type) {
    case 0:  // pivot: its tile after round r-1; pivot slot free (all panels of r-2 done)
      if (lane == 0) { p = ver + (size_t)k.r * R + k.r; target = k.r; return true; }
      if (lane == 1 && k.r >= 2) { p = a.done + (k.r - 2); target = 2 * (R - 1); return true; }
      return false;
    case 1:
    case 2:  // panel: its tile after round r-1, the pivot of r, snapshot slot free
      if (lane == 0) { p = ver + (size_t)k.ti * R + k.tj; target = k.r; return true; }
      if (lane == 1) { p = ver + (size_t)k.r * R + k.r; target = k.r + 1; return true; }
      if (lane == 2 && k.r >= 2) {
        p = a.done + R + (k.r - 2);
        target = (R - 1) * (R - 1);
        return true;
      }
      return false;
    default:  // remaining tile: itself after r-1, both panels of round r
      if (lane == 0) { p = ver + (size_t)k.ti * R + k.tj; target = k.r; return true; }
      if (lane == 1) { p = ver + (size_t)k.ti * R + k.r; target = k.r + 1; return true; }
      if (lane == 2) { p = ver + (size_t)k.r * R + k.tj; target = k.r + 1; return true; }
      // tile (r+1, r+1) fused with the pivot of round r+1: that pivot's
      // snapshot slot is free once every panel of round r-1 is done
      if (lane == 3 && k.type == kFusedTask && k.r >= 1) {
        p = a.done + (k.r - 1);
        target = 2 * (R - 1);
        return true;
      }
      return false;
  }
}

// Wait (bounded) until every input of task k exists: lane i of the producer
// warp acquires dependency i, so the waits overlap; the warp barrier then
// orders those acquires before the copies lane 0 issues.  Whole warp.
template <typename T>
__device__ bool wait_deps(const Args<T>& a, const fwh::Task& k, int lane) {
  const int* p = nullptr;
  int target = 0;
  bool ok = true;
  if (lane < 4 && dep_of(a, k, lane, p, target))
    ok = wait_ge(p, target, a.abort_flag, a.status, a.timeout_ns);
  return __all_sync(0xffffffffu, ok);
}

// Completion of task k: the tile's version, and the per-phase counters that
// guard snapshot slot reuse.  Release semantics make every store of the task
// (made by the compute warps and ordered before this thread through the
// task_done mbarrier) visible to whoever acquires the flag.
template <typename T>
__device__ __forceinline__ void publish(const Args<T>& a, const fwh::Task& k) {
  // (a fused task publishes its tile after round r+1's pivot: version r+2)
  st_release(a.ver + (size_t)k.ti * a.R + k.tj, k.type == kFusedTask ? k.r + 2 : k.r + 1);
  if (k.type == 1 || k.type == 2) red_release_add(reinterpret_cast<unsigned*>(a.done + k.r), 1u);
  if (k.type == 3 || k.type == kFusedTask)
    red_release_add(reinterpret_cast<unsigned*>(a.done + a.R + k.r), 1u);
}

// Copy the tile (k.ti, k.tj) of D into Dbuf (whole producer warp): one 2-D
// tensor copy, or one bulk copy per valid row.
template <typename T, int BS, int LBS>
__device__ __forceinline__ void issue_tile_load(const Args<T>& a, const fwh::Task& k,
                                                unsigned char* smem, WsBars* wb, PipeCnt& pc,
                                                int lane) {
  using L = WsLayout<LBS, T>;
  // the tile's own D block, one bulk copy per valid row
  const int64_t row0 = (int64_t)k.ti * BS, col0 = (int64_t)k.tj * BS;
  const int nrows = (int)(a.n - row0 < (int64_t)BS ? a.n - row0 : (int64_t)BS);
  const int ncols = (int)(a.n - col0 < (int64_t)BS ? a.n - col0 : (int64_t)BS);
  // whole 16-byte granules (rows are 16-byte aligned and ld % 4 == 0, so the
  // rounded row stays inside the caller's row)
  const unsigned rowbytes = (unsigned)(((size_t)ncols * sizeof(T) + 15) / 16 * 16);
  unsigned char* dbuf = smem + L::d_off();
  if (a.tmapD) {
    // one tensor copy of the whole box (elements beyond n arrive as zeros and
    // are masked by the compute warps); a single instruction keeps the
    // producer's issue slots, shared with two compute warps, free
    if (lane == 0) {
      if (!pc.stop && mbar_wait(&wb->d_empty, (pc.d & 1) ^ 1, a.status, a.abort_flag, a.timeout_ns)) {
        mbar_expect_tx(&wb->d_full, (unsigned)(BS * BS * sizeof(T)));
        tma_load_2d(dbuf, a.tmapD, (int)col0, (int)row0, &wb->d_full);
        pc.d_armed = pc.d + 1;
      } else {
        pc.stop = true;
      }
    }
  } else {
    bool ok = false;
    if (lane == 0) {
      ok = !pc.stop && mbar_wait(&wb->d_empty, (pc.d & 1) ^ 1, a.status, a.abort_flag, a.timeout_ns);
      if (ok) {
        mbar_expect_tx(&wb->d_full, rowbytes * (unsigned)nrows);
        pc.d_armed = pc.d + 1;
      } else {
        pc.stop = true;
      }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (ok)
      for (int rr = lane; rr < nrows; rr += 32)
        bulk_g2s(dbuf + (size_t)rr * BS * sizeof(T), a.D + (row0 + rr) * a.ld + col0, rowbytes,
                 &wb->d_full);
  }
  ++pc.d;
}

// How a remaining-tile task relaxes (mode) and the forms of its operands (kForm*).
// int32: over 16-bit keys when the sums of its panel tiles fit (mode: their
// clamp), else over 32-bit keys when those fit (1), else with compare and select
// (0; or packed keys off).  Unless mode > 1 an operand kept in 16 bits, or in
// exact 32-bit keys where values are wanted, is expanded by the compute warps.
// The other types: 0, or 2 where tiles are filtered by 16-bit bounds.  (The two
// bounds are loaded once, together: a second round trip to L2 would lie on the
// producer's serial path, which bounds small tiles.)
struct TileForm {
  int mode, dec;
};
template <typename T, int BS>
__device__ __forceinline__ TileForm tile_form(const Args<T>& a, const fwh::Task& k) {
  if (!Num<T>::kPacked) return {kFiltered<T, BS> ? 2 : 0, 0};
  if (!(a.packed && (k.type == 3 || k.type == kFusedTask))) return {0, 0};
  const int slot = k.r & 1;
  const int ba = __ldcg(a.colB + (size_t)slot * a.slot_tiles + k.ti);
  const int bb = __ldcg(a.rowB + (size_t)slot * a.slot_tiles + k.tj);
  if (const int cap = h_clamp<BS>(ba, bb)) return {cap, 0};
  const int mode = bnd_value(ba) + bnd_value(bb) < Keys<BS>::CAP ? 1 : 0;
  int form = ((ba & kBndInf) ? kFormInfA : 0) | ((bb & kBndInf) ? kFormInfB : 0);
  if (!(ba & kBndK)) form |= kFormHA;  // (16-bit keys only)
  else if (mode == 0 && bnd_value(ba) < Keys<BS>::CAP) form |= kFormKA;
  if (!(bb & kBndK)) form |= kFormHB;
  else if (mode == 0 && bnd_value(bb) < Keys<BS>::CAP) form |= kFormKB;
  return {mode, form};
}

// Issue the operand copies of remaining-tile task k (whole producer warp).
template <typename T, int BS, int LBS>
__device__ void issue_operands(const Args<T>& a, const fwh::Task& k, int mode, int dec,
                               unsigned char* smem, WsBars* wb, PipeCnt& pc, int lane) {
  using L = WsLayout<LBS, T>;
  using C = WsChunk<BS, T>;
  fence_proxy_async();  // global data published by other CTAs, read by TMA below
  const int slot = k.r & 1;
  const size_t toffA = ((size_t)slot * a.slot_tiles + k.ti) * BS * BS;
  const size_t toffB = ((size_t)slot * a.slot_tiles + k.tj) * BS * BS;
  if (mode > 1) {
    // 16-bit keys: both whole operand tiles in one stage; the tile itself is
    // needed after the relaxation only (its buffer may still be in use)
    constexpr unsigned bytes = BS * BS * 2;
    if (lane == 0) {
      const unsigned st = pc.chunk & 1;
      if (!pc.stop && mbar_wait(&wb->chunk_empty[st], ((pc.chunk >> 1) & 1) ^ 1, a.status,
                                a.abort_flag, a.timeout_ns)) {
        mbar_expect_tx(&wb->chunk_full[st], 2 * bytes);
        unsigned char* dst = smem + L::ring_off() + st * L::kStage;
        bulk_g2s(dst, a.colH + toffA / 2, bytes, &wb->chunk_full[st]);
        bulk_g2s(dst + bytes, a.rowH + toffB / 2, bytes, &wb->chunk_full[st]);
        pc.chunk_armed[st] = pc.chunk + 1;
      } else {
        pc.stop = true;
      }
    }
    ++pc.chunk;
    issue_tile_load<T, BS, LBS>(a, k, smem, wb, pc, lane);
    return;
  }
  if constexpr (kFiltered<T, BS>) return;
  constexpr bool kTileFirst = !std::is_same<T, float>::value;
  if (kTileFirst) issue_tile_load<T, BS, LBS>(a, k, smem, wb, pc, lane);
  // operand chunks
  const unsigned char* srcA = (mode || (dec & kFormKA)) ? (const unsigned char*)(a.colK + toffA)
                                                       : (const unsigned char*)(a.colR + toffA);
  const unsigned char* srcB = (mode || (dec & kFormKB)) ? (const unsigned char*)(a.rowK + toffB)
                                                       : (const unsigned char*)(a.rowR + toffB);
  // (a 16-bit tile comes whole with every chunk, which expands its part of it)
  unsigned bytesA = (unsigned)C::kChunkBytes, bytesB = bytesA;
  size_t stepA = C::kChunkBytes, stepB = stepA;
  if constexpr (Num<T>::kPacked) {
    static_assert((size_t)BS * BS * 2 <= C::kChunkBytes, "a 16-bit tile per operand chunk");
    if (dec & kFormHA) {
      srcA = (const unsigned char*)(a.colH + toffA / 2);
      bytesA = BS * BS * 2;
      stepA = 0;
    }
    if (dec & kFormHB) {
      srcB = (const unsigned char*)(a.rowH + toffB / 2);
      bytesB = BS * BS * 2;
      stepB = 0;
    }
  }
  // floating types, small tiles: the predecessors of the B panel's rows as well
  const unsigned bytesP = kPredSmem<T, BS> && a.P ? BS * BS * 4u : 0u;
  for (int c = 0; c < C::NC; ++c) {
    if (lane == 0) {
      const unsigned st = pc.chunk & 1;
      if (!pc.stop && mbar_wait(&wb->chunk_empty[st], ((pc.chunk >> 1) & 1) ^ 1, a.status,
                                a.abort_flag, a.timeout_ns)) {
        mbar_expect_tx(&wb->chunk_full[st], bytesA + bytesB + bytesP);
        unsigned char* dst = smem + L::ring_off() + st * L::kStage;
        bulk_g2s(dst, srcA + c * stepA, bytesA, &wb->chunk_full[st]);
        bulk_g2s(dst + C::kChunkBytes, srcB + c * stepB, bytesB, &wb->chunk_full[st]);
        if (bytesP) bulk_g2s(dst + 2 * C::kChunkBytes, a.rowP + toffB, bytesP, &wb->chunk_full[st]);
        pc.chunk_armed[st] = pc.chunk + 1;
      } else {
        pc.stop = true;
      }
    }
    ++pc.chunk;
  }
  // (fp32 reads the tile after the relaxation: its buffer may still be in use)
  if (!kTileFirst) issue_tile_load<T, BS, LBS>(a, k, smem, wb, pc, lane);
}

// Issue the operands of panel task k (whole producer warp): the tile into Dbuf,
// the closed pivot of round k.r into the next ring stage, and the stage after
// it handed over empty as the task's scratch (ws_panel, ws_panel_f).
template <typename T, int BS, int LBS>
__device__ void issue_panel_operands(const Args<T>& a, const fwh::Task& k, unsigned char* smem,
                                     WsBars* wb, PipeCnt& pc, int lane) {
  using L = WsLayout<LBS, T>;
  using C = WsChunk<BS, T>;
  fence_proxy_async();  // global data published by other CTAs, read by TMA below
  issue_tile_load<T, BS, LBS>(a, k, smem, wb, pc, lane);
  if (lane == 0) {
    const unsigned st = pc.chunk & 1;
    if (!pc.stop && mbar_wait(&wb->chunk_empty[st], ((pc.chunk >> 1) & 1) ^ 1, a.status,
                              a.abort_flag, a.timeout_ns)) {
      // fp32, small column panels: the pivot's predecessors as well
      const unsigned bytesP = kPredSmem<T, BS> && a.P && k.type == 2 ? BS * BS * 4u : 0u;
      mbar_expect_tx(&wb->chunk_full[st], (unsigned)C::kTile + bytesP);
      unsigned char* const dst = smem + L::ring_off() + st * L::kStage;
      bulk_g2s(dst, a.piv + (size_t)(k.r & 1) * BS * BS, (unsigned)C::kTile, &wb->chunk_full[st]);
      if (bytesP)
        bulk_g2s(dst + C::kTile, a.pivP + (size_t)(k.r & 1) * BS * BS, bytesP, &wb->chunk_full[st]);
      pc.chunk_armed[st] = pc.chunk + 1;
    } else {
      pc.stop = true;
    }
    const unsigned st1 = (pc.chunk + 1) & 1;
    if (!pc.stop && mbar_wait(&wb->chunk_empty[st1], (((pc.chunk + 1) >> 1) & 1) ^ 1, a.status,
                              a.abort_flag, a.timeout_ns)) {
      mbar_arrive(&wb->chunk_full[st1]);  // no copy: the stage is scratch
      // (recorded all the same: the final drain waits on the latest phase of
      // each barrier, and a parity wait on an older one would never succeed
      // once the barrier is two phases further)
      pc.chunk_armed[st1] = pc.chunk + 2;
    } else {
      pc.stop = true;
    }
  }
  pc.chunk += 2;
}

// Optional per-task trace (sampled tasks): 10 words per entry.
//   [0] task | type << 32 | graph << 40   [1] SM id
//   producer: [2] claimed  [3] inputs ready  [4] copies issued  [5] published
//   compute : [6] descriptor seen  [9] task finished (stores issued)
//   min-plus tasks: [7], [8] SM-cycle counts of the task's phases
__device__ __forceinline__ uint64_t* trace_slot(uint64_t* tr, int cap, int stride, int64_t t) {
  if (!tr || t < 0 || stride <= 0 || t % stride) return nullptr;
  const int64_t s = t / stride;
  return s < cap ? tr + (size_t)s * 10 : nullptr;
}
__device__ __forceinline__ unsigned smid() {
  unsigned r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return r;
}

// Runs f(std::integral_constant<int, BS>) for the block size of the task.
// kFixedBS > 0: that block size only (single-graph kernels).
template <int kFixedBS, int LBS, typename F>
__device__ __forceinline__ auto with_bs(int bs, F&& f) {
  if constexpr (kFixedBS > 0) {
    return f(std::integral_constant<int, kFixedBS>{});
  } else {
    if (bs == 32) return f(std::integral_constant<int, 32>{});
    if constexpr (LBS >= 64)
      if (bs == 64) return f(std::integral_constant<int, 64>{});
    return f(std::integral_constant<int, LBS>{});
  }
}

// ------------------------------------------------------------------ engine ----

// Src supplies: total(), next (claim counter), status / abort / timeout, trace,
// resolve(t, &g) -> local task, args(g) -> const Args<T>&, bs(g).
template <typename T, int kFixedBS, int LBS, class Src>
__device__ void ws_engine(const Src& src, unsigned char* smem, WsBars& wb, CtaScratch& cs) {
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&wb.desc_full[i], 1);
      mbar_init(&wb.desc_empty[i], kThreads / 32);
      mbar_init(&wb.chunk_full[i], 1);
      mbar_init(&wb.chunk_empty[i], kThreads / 32);
    }
    mbar_init(&wb.d_full, 1);
    mbar_init(&wb.d_empty, kThreads / 32);
    for (int i = 0; i < kPubDepth; ++i) {
      mbar_init(&wb.pub_full[i], 1);
      mbar_init(&wb.pub_empty[i], 1);
      mbar_init(&wb.task_done[i], kThreads / 32);
      wb.pst[i] = 0;
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == kThreads / 32 + 1) {
    // ----------------------------------------------------------- publisher
    // One lane waits and publishes: with the whole warp in step on every wait a
    // publication came 0.35 us later, three times a round on the chain that
    // bounds small solves (n = 1000, int64: 1.35 -> 1.39 ms).  The other lanes
    // join for the copies of a 16-bit panel.
    unsigned i = 0;
    auto finish = [&](unsigned q, int t, const fwh::Task& k, int g) {
      if (t != src.skip_task) publish(src.args(g), k);
      if (uint64_t* tr = trace_slot(src.trace, src.trace_cap, src.trace_stride, t))
        tr[5] = globaltimer();
      mbar_arrive(&wb.pub_empty[q]);
    };
    for (;;) {
      int pst = 0;
      if (lane == 0) {
        for (;; ++i) {
          const unsigned q = i % kPubDepth, ph = (i / kPubDepth) & 1;
          if (!mbar_wait(&wb.pub_full[q], ph, src.status, src.abort_flag, src.timeout_ns)) break;
          const int t = wb.pubq[q][0];
          const fwh::Task k{wb.pubq[q][1], wb.pubq[q][2], wb.pubq[q][3], wb.pubq[q][4]};
          const int g = wb.pubq[q][5];
          if (t < 0) break;
          // tasks finish in hand-off order: the i-th completion is this task
          if (!mbar_wait(&wb.task_done[q], ph, src.status, src.abort_flag, src.timeout_ns)) break;
          if constexpr (Num<T>::kPacked) {
            if ((k.type == 1 || k.type == 2) && (wb.pst[q] & kPstOn)) {
              pst = wb.pst[q];
              break;
            }
          }
          finish(q, t, k, g);
        }
      }
      if constexpr (!Num<T>::kPacked) {
        break;
      } else {
        pst = __shfl_sync(0xffffffffu, pst, 0);
        i = __shfl_sync(0xffffffffu, i, 0);
        __syncwarp();
        if (!pst) break;
        const unsigned q = i % kPubDepth;
        const fwh::Task k{wb.pubq[q][1], wb.pubq[q][2], wb.pubq[q][3], wb.pubq[q][4]};
        const int t = wb.pubq[q][0], g = wb.pubq[q][5];
        with_bs<kFixedBS, LBS>(src.bs(g), [&](auto B) {
          store_panel<T, decltype(B)::value, LBS>(src.args(g), k, pst, smem, &wb, lane);
          return 0;
        });
        if (lane == 0) finish(q, t, k, g);
        ++i;
        __syncwarp();
      }
    }
    return;
  }

  if (warp == kThreads / 32) {
    // ------------------------------------------------------------ producer
    constexpr bool own_panels = kFixedBS > 0 && kOwnPanels<T, kFixedBS>;  // (batches: 32-bit types)
    const int64_t total = src.total();
    unsigned idesc = 0, ipub = 0;
    PipeCnt pc;
    for (;;) {
      int t = -1, g = 0;
      uint64_t t_claim = 0;
      if (lane == 0) {
        t_claim = globaltimer();
        const int ab = ld_relaxed(src.abort_flag);  // (in flight together with the claim)
        const int64_t tt = atomicAdd(src.next, 1u);
        if (tt < total && !ab) t = (int)tt;
      }
      // lane 0 decodes the task; the others take it by shuffle
      fwh::Task k{0, 0, 0, 0};
      if (lane == 0 && t >= 0) k = src.resolve(t, g);
      t = __shfl_sync(0xffffffffu, t, 0);
      g = __shfl_sync(0xffffffffu, g, 0);
      k.type = __shfl_sync(0xffffffffu, k.type, 0);
      k.r = __shfl_sync(0xffffffffu, k.r, 0);
      k.ti = __shfl_sync(0xffffffffu, k.ti, 0);
      k.tj = __shfl_sync(0xffffffffu, k.tj, 0);
      if (t >= 0) {
        // tile (r+1, r+1) of round r takes the pivot of round r+1 along, and
        // that pivot's own queue entry is skipped
        if (k.type == 0 && k.r >= 1) continue;
        if (k.type == 3 && k.ti == k.r + 1 && k.tj == k.r + 1) k.type = kFusedTask;
        if (!wait_deps(src.args(g), k, lane)) t = -1;
      }
      if (lane == 0) {
        if (uint64_t* tr = trace_slot(src.trace, src.trace_cap, src.trace_stride, t)) {
          tr[1] = smid();
          tr[2] = t_claim;
          tr[3] = globaltimer();
        }
      }
      int mode = 0;
      int dec = 0;
      int bs = 0;
      if (t >= 0) {
        bs = src.bs(g);
        const TileForm form = with_bs<kFixedBS, LBS>(
            bs, [&](auto B) { return tile_form<T, decltype(B)::value>(src.args(g), k); });
        mode = form.mode;
        dec = form.dec;
      }
      unsigned pq = 0;
      if (lane == 0) {
        // queue the task for publication, then hand it to the compute warps
        pq = ipub % kPubDepth;
        mbar_wait(&wb.pub_empty[pq], ((ipub / kPubDepth) & 1) ^ 1, src.status, src.abort_flag,
                  src.timeout_ns);
        wb.pubq[pq][0] = t;
        wb.pubq[pq][1] = k.type;
        wb.pubq[pq][2] = k.r;
        wb.pubq[pq][3] = k.ti;
        wb.pubq[pq][4] = k.tj;
        wb.pubq[pq][5] = g;
        mbar_arrive(&wb.pub_full[pq]);
        const unsigned ds = idesc & 1;
        mbar_wait(&wb.desc_empty[ds], ((idesc >> 1) & 1) ^ 1, src.status, src.abort_flag,
                  src.timeout_ns);
        wb.desc[ds][0] = t;
        wb.desc[ds][1] = k.type;
        wb.desc[ds][2] = k.r;
        wb.desc[ds][3] = k.ti;
        wb.desc[ds][4] = k.tj;
        wb.desc[ds][5] = mode;
        wb.desc[ds][6] = g;
        wb.desc[ds][7] = dec;
        mbar_arrive(&wb.desc_full[ds]);
      }
      ++idesc;
      ++ipub;
      if (t < 0) break;
      if (k.type == 3 || k.type == kFusedTask) {
        with_bs<kFixedBS, LBS>(bs, [&](auto B) {
          issue_operands<T, decltype(B)::value, LBS>(src.args(g), k, mode, dec, smem, &wb, pc,
                                                     lane);
          return 0;
        });
        if (k.type == kFusedTask && lane == 0) {
          // its pivot uses the shared buffer as scratch: wait until the task
          // has been published (its publication-queue slot frees up)
          mbar_wait(&wb.pub_empty[pq], (((ipub - 1) / kPubDepth) & 1), src.status,
                    src.abort_flag, src.timeout_ns);
        }
      } else if (k.type != 0 && !own_panels) {
        with_bs<kFixedBS, LBS>(bs, [&](auto B) {
          if constexpr (!own_panels)
            issue_panel_operands<T, decltype(B)::value, LBS>(src.args(g), k, smem, &wb, pc, lane);
          return 0;
        });
      } else {
        if (lane == 0) {
          // the task uses the shared buffer as scratch: wait until it has been
          // published (its publication-queue slot frees up)
          mbar_wait(&wb.pub_empty[pq], (((ipub - 1) / kPubDepth) & 1), src.status,
                    src.abort_flag, src.timeout_ns);
        }
      }
      if (lane == 0) {
        if (uint64_t* tr = trace_slot(src.trace, src.trace_cap, src.trace_stride, t)) {
          tr[0] = (uint64_t)(unsigned)t | ((uint64_t)k.type << 32) | ((uint64_t)(unsigned)g << 40);
          tr[4] = globaltimer();
        }
      }
      if (k.type == 0 || k.type == kFusedTask || (own_panels && k.type != 3)) fence_proxy_async();
      __syncwarp();
    }
    // leave no bulk copy in flight: wait for the last phase armed with a copy on
    // every full barrier
    if (lane == 0) {
      if (pc.d_armed)
        mbar_wait(&wb.d_full, (pc.d_armed - 1) & 1, src.status, src.abort_flag, src.timeout_ns);
      for (int st = 0; st < 2; ++st)
        if (pc.chunk_armed[st])
          mbar_wait(&wb.chunk_full[st], ((pc.chunk_armed[st] - 1) >> 1) & 1, src.status,
                    src.abort_flag, src.timeout_ns);
    }
    return;
  }

  // -------------------------------------------------------------- compute
  if (warp >= kThreads / 64) turn_pass(0);  // group 0 has the first turn
  unsigned idesc = 0;
  PipeCnt pc;
  for (;;) {
    const unsigned ds = idesc & 1;
    if (!mbar_wait(&wb.desc_full[ds], (idesc >> 1) & 1, src.status, src.abort_flag,
                   src.timeout_ns))
      break;
    const int t = wb.desc[ds][0];
    const fwh::Task k{wb.desc[ds][1], wb.desc[ds][2], wb.desc[ds][3], wb.desc[ds][4]};
    const int mode = wb.desc[ds][5];
    const int g = wb.desc[ds][6];
    const int dec = wb.desc[ds][7];
    __syncwarp();
    if (lane == 0) mbar_arrive(&wb.desc_empty[ds]);
    ++idesc;
    if (t < 0) break;
    uint64_t* tr = tid == 0 ? trace_slot(src.trace, src.trace_cap, src.trace_stride, t) : nullptr;
    if (tr) tr[6] = globaltimer();
    const bool ok = with_bs<kFixedBS, LBS>(src.bs(g), [&](auto B) {
      return compute_task<T, decltype(B)::value, LBS>(src.args(g), k, mode, dec, smem, &wb, &cs,
                                                      pc, (idesc - 1) % kPubDepth, tr);
    });
    if (tr) tr[9] = globaltimer();
    if (!ok) break;
    __syncwarp();
    if (lane == 0) mbar_arrive(&wb.task_done[(idesc - 1) % kPubDepth]);
  }
}

// One graph: the queue of decode_task, block size BS.  `a` lies in shared memory:
// as a local copy per thread (the tensor-map pointers are filled in here) its
// lines took most of the L1 cache that 226 KB of shared memory leave, and many a
// pointer or size that a task reads came from L2 (panels of 128: 2 to 3 K of 92 K
// cycles).
template <typename T, int BS>
struct SingleSrc {
  const Args<T>& a;
  unsigned* next;
  int* status;
  int* abort_flag;
  int64_t timeout_ns;
  int skip_task;
  uint64_t* trace;
  int trace_cap, trace_stride;
  int R;
  int64_t lookahead;
  const unsigned* stage_off;
  mutable int stage = 0;   // of the latest task that resolve decoded
  __device__ SingleSrc(const Args<T>& x, const Args<T>& shared)
      : a(shared), next(x.ctr), status(x.status), abort_flag(x.abort_flag),
        timeout_ns(x.timeout_ns), skip_task(x.skip_task), trace(x.trace),
        trace_cap(x.trace_cap), trace_stride(x.trace_stride), R(x.R), lookahead(x.lookahead),
        stage_off(x.stage_off) {}
  __device__ int64_t total() const { return stage_off[R + 1]; }
  __device__ fwh::Task resolve(int64_t t, int& g) const {
    g = 0;
    return fwh::decode_task(t, R, lookahead, stage_off, stage);
  }
  __device__ const Args<T>& args(int) const { return a; }
  __device__ int bs(int) const { return BS; }
};

template <typename T, int BS, int kCtas>
__global__ void __launch_bounds__(kWsThreads, kCtas)
    k_persistent_ws(Args<T> a, const __grid_constant__ CUtensorMap tmD,
                    const __grid_constant__ CUtensorMap tmP, int use_tmap) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ WsBars wb;
  __shared__ CtaScratch cs;
  // use_tmap: bit 0 the D map, bit 1 the P map
  __shared__ Args<T> args;
  if (threadIdx.x == 0) {
    args = a;
    args.tmapD = (use_tmap & 1) ? &tmD : nullptr;
    args.tmapP = (use_tmap & 2) ? &tmP : nullptr;
  }
  // (ws_engine's first barrier precedes every use)
  const SingleSrc<T, BS> src(a, args);
  ws_engine<T, BS, BS>(src, smem, wb, cs);
}

// The kernel for R x R tiles, by CTAs per SM.  Filtered fp64: two (96 registers
// per thread), so that the gathers of one's exact relaxations overlap the other's
// work, from five tiles per SM and round on.  With fewer, tiles and the chain of
// pivots would share an SM's narrow FP64 pipe while other SMs are idle (two / one
// CTA per SM, uniform n = 700 2.47 / 2.02 ms, n = 1100 3.58 / 3.02, n = 1650 5.12 /
// 4.57, n = 1800 5.70 / 5.33; a far vertex in each block n = 900 4.1 / 3.7, n = 1350
// 6.1 / 5.7, n = 1650 7.6 / 9.2, n = 1800 8.6 / 11.7).
// Tiles of 64 with 32-bit elements: a tile is done in 2.7 us (int32, 16-bit
// keys) to 7 us (fp32), in which a lone CTA waits for its operands half of the
// time; two overlap that, but also share the SM with the tasks that the chain of
// pivots waits for.  From 12 tiles per SM and round on the first counts more (one /
// two CTAs per SM, int32 R = 36 1.34 / 1.42 ms, R = 41 1.83 / 1.77, R = 47 2.62 /
// 2.22; weights to 3e5, R = 41 1.91 / 1.92, R = 47 2.75 / 2.60; fp32 R = 36 2.15 /
// 2.17, R = 41 3.04 / 2.79, R = 47 4.53 / 4.26).  Two CTAs leave a thread 96
// registers; the kernel for one uses 129 (int32) or 134 (fp32), and at 96 it is 2 %
// slower (n = 1000 0.60 -> 0.61 ms).
template <typename T, int BS>
auto persistent_kernel(int R) {
  if constexpr (BS == 64 && sizeof(T) == 4)
    if ((int64_t)R * R >= 12 * (int64_t)fwh::num_sms()) return k_persistent_ws<T, BS, 2>;
  if constexpr (kFiltered<T, BS>)
    if ((int64_t)R * R > 5 * (int64_t)fwh::num_sms()) return k_persistent_ws<T, BS, 2>;
  return k_persistent_ws<T, BS, 1>;
}

}  // namespace fwk
