// The history convolution blocked in time (Section 2.3, the per-mode truncated
// time convolution of s_i), for float-class histories.
//
// One step alone has to read every mode's whole history: 24 bytes per mode and
// lag for 10 multiply-adds, 1.05 of the copy bandwidth and 1/14 of the FP32 rate
// when it is done step by step.  Consecutive steps read the same history, though,
// so the sums are blocked in time: from the history before a block's first step
// `base`, one pass (ahead_kernel) forms the sums of the block's kAhead = 16 steps,
//     A[s] = sum_{m >= 1} w(m + s) D[base - m],   s = 0 .. 15,
// and each step of the block adds the at most 16 lags that lie inside the block
// (near_kernel).  The history is read once per 16 steps and the work per step is
// the same multiply-adds, now bound by the FP32 pipe (39-40 T multiply-adds/s
// measured on GB300: 0.54 ms for 1024^2 x 4096 against 7.1 ms for the bytes).  The kernel
// takes 1.11 ms there, ~155 ns per lag of a CTA against 77 on the pipe alone: 16 of a
// warp's 33 instructions per lag are the two-lane multiply-adds and 2 the folds (ncu,
// 512^2 x 1024), and the pipe is busy 59 % of the time.  A warp set aside for the
// requests (spills: 21 warps leave 80 registers), the requests in turns behind an
// mbarrier (+3 %), a skew of at most one (+15 %) or two stages (+1 %) between the warps,
// and weights loaded into both halves of a register pair (same) were measured and not kept.
//
// Blocks are aligned and staggered: tile T (128 records) starts its blocks at the
// steps with (n + T) mod 16 = 0, so every step of a plane of 16 and more tiles renews
// about 1/16 of them and costs the same (smaller planes have steps that renew none).
// A tile's block is a function of n and T only, and every sum has a fixed order, so a
// step's result does not depend on when its sums were formed: a restored checkpoint, a
// rewound or repeated step and a replayed graph give the same bits as the run they
// continue.  Each (chunk, tile, 32 records) carries a stamp
// of the block its sums belong to and of the arguments' chunking and window; sums
// whose stamp is not the current one are formed again, all on the device, so that a
// captured graph renews them as a direct step does.  sbim_reset and sbim_load, which
// change the ring itself, mark every stamp invalid, and the second of two sbim_rewind
// calls in a row those of blocks that begin after the step it goes back to: a level
// before them may be written again, and a block whose predecessor has no history in a
// chunk finds its old stamp there.
#pragma once

#include <type_traits>

#include "../../include/sbim.h"
#include "sbim_conv_tma.cuh"
#include "sbim_device.cuh"

namespace sbim {
namespace ahead {

using namespace dev;

// 32 records x 4 members x 5 complex sums per CTA, one complex sum of one member per
// thread: 20 warps, one CTA per SM.  Warp k holds sum k / 4 of the records 8 (k % 4)
// .. + 7, so each of the SM's four schedulers has five warps and the same work (CTAs
// of 5 warps, 8 records, put two of them on the first scheduler each: 1.16 ms for
// 1024^2 x 4096 against 1.05, folding every 64 lags).  A thread keeps 16 outputs (32 registers) and a window
// of 16 weights, each held twice so that one two-lane multiply-add takes (re, im) (32
// registers).
constexpr int kRec = kAheadRec, kSums = 5, kThreads = kRec * kMembers * kSums, kWarps = kThreads / 32;
constexpr int kSub = kOrbitTile / kRec;     // CTAs per 128-record tile
constexpr int kLags = kAheadLags;   // lags per stage
constexpr int kFoldAll = 97;        // first lag of the longer chains
template <bool HALVES> __host__ __device__ constexpr int stages() { return HALVES ? 4 : 5; }

template <class S> __host__ __device__ constexpr int seg() { return kRec * S::kRecBytes; }
template <class S> __host__ __device__ constexpr int hist_bytes() { return kLags * 3 * S::kPlanes * seg<S>(); }
// The weights of one lag: 32 records (x 2 halves) x (11, 22, 33, 12).
template <bool HALVES> __host__ __device__ constexpr int wlag_bytes() { return (HALVES ? 2 : 1) * kRec * 16; }
// A stage: 8 lags of history and the weights 16 lags further on.
template <class S, bool HALVES> __host__ __device__ constexpr int stage_bytes() {
  return hist_bytes<S>() + kLags * wlag_bytes<HALVES>();
}
constexpr int kSumBytes = kThreads * kAhead * 8;   // the running sums
template <class S, bool HALVES> __host__ __device__ constexpr int smem_bytes() {
  return stages<HALVES>() * stage_bytes<S, HALVES>() + kSumBytes;
}
__device__ __forceinline__ unsigned long long fma2r(unsigned long long a, unsigned long long b,
                                                    unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long add2r(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long sub2r(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Counts one up and returns the value before: releases what this thread did, and the
// one that reads the last count sees what the others released.
__device__ __forceinline__ int shared_inc(int* p) {
  int r;
  asm volatile("atom.acq_rel.cta.shared.add.s32 %0, [%1], 1;" : "=r"(r) : "r"(tma::smem_addr(p)) : "memory");
  return r;
}
__device__ __forceinline__ void tile_g2s(unsigned dst, const void* map, int x, int y, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}

// One member's value: in a staged row (32 records; the lo plane `lo` bytes on), in
// the ring, and as stored.
template <class S> struct MemberIO;
template <> struct MemberIO<StoreF32> {
  __device__ static float2 smem(const unsigned char* p, int, int lane) {
    return *reinterpret_cast<const float2*>(p + lane * 8);
  }
  __device__ static float2 load(const void* h, long long i, long long) {
    return __ldcg(reinterpret_cast<const float2*>(h) + i);
  }
  __device__ static float2 store(void* h, long long i, long long, float2 d) {
    reinterpret_cast<float2*>(h)[i] = d;
    return d;
  }
};
template <bool LO> struct MemberIO<StoreBF16<LO>> {
  __device__ static float2 smem(const unsigned char* p, int lo, int lane) {
    float2 d = unpack_bf16(*reinterpret_cast<const unsigned*>(p + lane * 4));
    if (LO) {
      const float2 l = unpack_bf16(*reinterpret_cast<const unsigned*>(p + lo + lane * 4));
      d.x += l.x;
      d.y += l.y;
    }
    return d;
  }
  __device__ static float2 load(const void* h, long long i, long long plane) {
    const unsigned* p = reinterpret_cast<const unsigned*>(h) + i;
    float2 d = unpack_bf16(__ldcg(p));
    if (LO) {
      const float2 l = unpack_bf16(__ldcg(p + plane * 4));
      d.x += l.x;
      d.y += l.y;
    }
    return d;
  }
  // stores the rounded value and returns it as the convolution reads it back
  __device__ static float2 store(void* h, long long i, long long plane, float2 d) {
    unsigned* p = reinterpret_cast<unsigned*>(h) + i;
    const unsigned hw = pack_bf16(d.x, d.y);
    float2 r = unpack_bf16(hw);
    p[0] = hw;
    if (LO) {
      const unsigned lw = pack_bf16(d.x - r.x, d.y - r.y);
      p[plane * 4] = lw;
      const float2 l = unpack_bf16(lw);
      r.x += l.x;
      r.y += l.y;
    }
    return r;
  }
};

// First step of the block of 16 steps that holds step n, for tile T (may be
// negative at the start of a run, when the block's sums are empty).
__device__ __forceinline__ long long block_base(long long n, int T) {
  return n - ((n + T) & (kAhead - 1));
}
// The stamp of sums formed for a block with these arguments' chunking and window.
__device__ __forceinline__ long long block_mark(const StepArgs& a, long long base) {
  return stamp_of(base, a.config_id);
}
// Largest lag m of the block sums A[s] of tile T: the history before `base`, the
// cutoff, and the tile's truncation window.
__device__ __forceinline__ int last_lag(const StepArgs& a, long long base, int T) {
  int m = a.n_cut - 1;
  if (base < m) m = (int)(base < 0 ? 0 : base);
  if (a.tile_lmax) m = min(m, a.tile_lmax[T] - 1);
  return m;
}

// What one CTA sums at a time: records 32 q .. 32 q + 31 of tile T over the lags m0 ..
// m1 of a chunk, in blocks of 16 lags.
struct Item {
  int T, rec0, m0, m1, nblk, chunk, bs;
  long long base;
  __device__ void set(const StepArgs& a, int T_, int q, int chunk_, long long n) {
    T = T_;
    chunk = chunk_;
    base = block_base(n, T);
    rec0 = T * kOrbitTile + q * kRec;
    m0 = 1 + chunk * a.ahead_lc;
    m1 = min(m0 + a.ahead_lc - 1, last_lag(a, base, T));
    nblk = (m1 - m0 + kAhead) / kAhead;
    bs = base < 0x7fffffff ? (int)base % a.n_cut : (int)(base % a.n_cut);
  }
};

// Shared state of a CTA: copies landed per stage, warps that have left it, the stages
// requested so far, and the item (kept here: a request needs it, the sums do not).
struct Sync {
  unsigned long long full[5];
  int left[5];
  unsigned requested;
  Item it;
};

// Request stage j of an item, the CTA's g-th (one thread): the lags m0 + 8 j .. + 7 and
// the weights 16 lags on.  The history of 8 lags is 24 rows of the ring (slot x
// component, 32 records each) and arrives as one tiled copy per plane; only where the
// 8 slots wrap around the ring, row by row.  (Copying every row by itself took the
// issuing warp four times as many instructions as its sums: 1.96 against 1.42 ms for
// 1024^2 x 4096.)
template <class S, bool HALVES>
__device__ __forceinline__ void request_stage(const StepArgs& a, int j, unsigned g, unsigned char* smem,
                                           Sync& sync) {
  const Item& it = sync.it;
  constexpr int SEG = seg<S>(), PLANE = hist_bytes<S>() / S::kPlanes, WL = wlag_bytes<HALVES>();
  const int buf = (int)(g % stages<HALVES>());
  unsigned char* st = smem + buf * stage_bytes<S, HALVES>();
  const unsigned bar = tma::smem_addr(&sync.full[buf]), dst = tma::smem_addr(st);
  const int mb = it.m0 + j * kLags;
  int top = it.bs - mb;                          // slot of the stage's first lag
  if (top < 0) top += a.n_cut;
  const bool tiled = top >= kLags - 1;
  const int lags = max(0, min(kLags, it.m1 - mb + 1));
  tma::mbar_expect_tx(bar, kLags * WL + (tiled ? hist_bytes<S>() : lags * 3 * S::kPlanes * SEG));
  tma::bulk_g2s(dst + hist_bytes<S>(),
                a.wts32 + ((long long)(it.rec0 / kRec) * ahead_weight_lags(a.n_cut) + mb + kAhead) * WL,
                kLags * WL, bar);
  if (tiled) {
#pragma unroll
    for (int pl = 0; pl < S::kPlanes; ++pl)
      tile_g2s(dst + pl * PLANE, a.tmap, it.rec0 * (S::kRecBytes / 4),
               (pl * a.n_cut + top - (kLags - 1)) * 3, bar);
  } else {
    const unsigned char* hist = reinterpret_cast<const unsigned char*>(a.hist);
    for (int i = 0; i < lags * 3 * S::kPlanes; ++i) {
      const int pl = i % S::kPlanes, l = i / S::kPlanes / 3, c = i / S::kPlanes % 3;
      int slot = top - l;
      if (slot < 0) slot += a.n_cut;
      tma::bulk_g2s(dst + pl * PLANE + ((kLags - 1 - l) * 3 + c) * SEG,
                    hist + (pl * a.slot_stride + ((long long)slot * 3 + c) * a.n_orb_pad + it.rec0) *
                               S::kRecBytes,
                    SEG, bar);
    }
  }
}

// A warp's part of an item: one of the five sums for the 32 members of 8 records.
// The terms of 16 lags (32 from lag kFoldAll on) are chained by multiply-adds, then
// folded into the running sums (in shared memory) with one compensated addition.  With
// chains of 32 lags throughout, and float weights inside the block, the error against 64
// bits was up to 0.6 % above that of the step-by-step convolution (compensated every 2
// lags); with 16 for the lags that carry the largest weights, and the stored weights
// inside the block, it is 0.99 of it for FP32 on average and equal for BF16 hi/lo (36
// sizes, spectra and precisions).  Chains of 16 throughout gain 0.1 % more and cost 4 %
// of a step (512^2 x 2000: 206 against 215 us), of 8 lags 18 %.  The warps meet only at
// the stages: each waits for its copies, and the last to leave one requests its next
// filling.  Returns false if a bounded wait gave up.
template <class S, bool HALVES>
__device__ __forceinline__ bool sum_item(const StepArgs& a, int q, unsigned char* smem, Sync& sync,
                                         unsigned g) {
  const Item& it = sync.it;
  const int m0 = it.m0, m1 = it.m1, nblk = it.nblk, n_cut = a.n_cut;
  constexpr int SEG = seg<S>(), STAGE = stage_bytes<S, HALVES>(), PLANE = hist_bytes<S>() / S::kPlanes;
  constexpr int WL = wlag_bytes<HALVES>(), NS = stages<HALVES>();
  using IO = MemberIO<S>;
  using u64 = unsigned long long;
  const int tid = threadIdx.x, lane = tid & 31;
  const int f = tid / kOrbitTile, x = tid % kOrbitTile;      // the sum (C11, C33, C22, C12a, C12b); member
  const int comp = f == 0 || f == 4 ? 0 : (f == 1 ? 2 : 1);
  const int kern = f == 0 ? 0 : (f == 1 ? 2 : (f == 2 ? 1 : 3));
  const int woff = (HALVES ? x >> 1 : x >> 2) * 16 + kern * 4;
  // lags with a weight: the cutoff's zeros are in the weights, a window's are not
  const int lim = a.lmax ? a.lmax[2 * (it.rec0 + (x >> 2)) + ((x >> 1) & 1)] : 0x7fffffff;
  // this thread's running sums, two per 16 bytes, strided over the threads
  ulonglong2* run = reinterpret_cast<ulonglong2*>(smem + NS * STAGE) + tid;

  u64 y[kAhead], w[kAhead];
  {
    const unsigned char* w0 = a.wts32 + ((long long)(it.rec0 / kRec) * ahead_weight_lags(a.n_cut) + it.m0) * WL + woff;
#pragma unroll
    for (int s = 0; s < kAhead; ++s) {
      y[s] = 0ull;                               // (0.f, 0.f)
      float v = __ldg(reinterpret_cast<const float*>(w0 + s * WL));
      if (it.m0 + s >= lim) v = 0.f;
      w[s] = pack2(make_float2(v, v));
      if (s % 2) run[(s / 2) * kThreads] = make_ulonglong2(0ull, 0ull);
    }
  }
  for (int b = 0; b < nblk; ++b) {
    const int mb = m0 + b * kAhead;
    bool ok = true;
    // Half a block, one stage: at lag l output s takes weight l + s of the window;
    // slot l is then replaced by the weight 16 lags on.
    auto half = [&](auto first, auto tail, auto window) {
      constexpr bool TAIL = decltype(tail)::value;
      constexpr int L0 = decltype(first)::value;
      const int buf = (int)(g % NS);
      ok = __all_sync(0xffffffffu, tma::mbar_wait(tma::smem_addr(&sync.full[buf]), (g / NS) & 1u, a.err));
      if (!ok) return;
      const unsigned char* st = smem + buf * STAGE;
      float2 dn = IO::smem(st + ((kLags - 1) * 3 + comp) * SEG, PLANE, x);
#pragma unroll
      for (int k = 0; k < kLags; ++k) {
        const int l = L0 + k;
        float2 d = dn;                           // the next lag's value is on its way
        if (k + 1 < kLags) dn = IO::smem(st + ((kLags - 2 - k) * 3 + comp) * SEG, PLANE, x);
        if (TAIL && mb + l > m1) d = make_float2(0.f, 0.f);
        const u64 dd = pack2(d);
        float v = *reinterpret_cast<const float*>(st + hist_bytes<S>() + woff + k * WL);
        if (decltype(window)::value && mb + kAhead + l >= lim) v = 0.f;
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
          // terms past the cutoff are left out, not multiplied by zero: a
          // non-finite value leaves the sums with its last lag
          const u64 ds = TAIL && mb + l + s >= n_cut ? 0ull : dd;
          y[s] = fma2r(w[(l + s) % kAhead], ds, y[s]);
        }
        w[l] = pack2(make_float2(v, v));
      }
      __syncwarp();
      if (lane == 0) {
        const int j = 2 * b + L0 / kLags;
        if (shared_inc(&sync.left[buf]) % kWarps == kWarps - 1 && j + NS < 2 * nblk) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          sync.requested = g + NS + 1;
          request_stage<S, HALVES>(a, j + NS, g + NS, smem, sync);
        }
      }
      ++g;
    };
    using Lo = std::integral_constant<int, 0>;
    using Hi = std::integral_constant<int, kLags>;
    auto block = [&](auto tail, auto window) {
      half(Lo{}, tail, window);
      if (ok) half(Hi{}, tail, window);
    };
    if (mb + 2 * kAhead - 2 >= n_cut || mb + kAhead - 1 > m1)
      block(std::true_type{}, std::true_type{});
    else if (a.lmax)
      block(std::false_type{}, std::true_type{});
    else
      block(std::false_type{}, std::false_type{});
    if (!ok) return false;
    if (b % 2 || mb < kFoldAll) {
#pragma unroll
      for (int s = 0; s < kAhead; s += 2) {
        const ulonglong2 o = run[(s / 2) * kThreads];
        const ulonglong2 t = make_ulonglong2(add2r(o.x, y[s]), add2r(o.y, y[s + 1]));
        y[s] = sub2r(y[s], sub2r(t.x, o.x));     // minus the compensation
        y[s + 1] = sub2r(y[s + 1], sub2r(t.y, o.y));
        run[(s / 2) * kThreads] = t;
      }
    }
  }
  float* out = a.ahead + (((long long)it.chunk * (a.n_orb_pad / kOrbitTile) + it.T) * kAhead * kFields + 2 * f) *
                             (kOrbitTile * kMembers) + q * (kRec * kMembers) + x;
#pragma unroll
  for (int s = 0; s < kAhead; ++s) {
    const ulonglong2 o2 = run[(s / 2) * kThreads];
    const float2 r = unpack2(add2r(s % 2 ? o2.y : o2.x, y[s]));
    float* o = out + (long long)s * kFields * (kOrbitTile * kMembers);
    o[0] = r.x;
    o[kOrbitTile * kMembers] = r.y;
  }
  return true;
}

// The tiles 16 i .. 16 i + 15 of one update, records 32 q .. of each, one chunk of
// lags: in a running time loop one of the 16 starts a new block at every step.
template <class S, bool HALVES>
__device__ __forceinline__ void ahead_tiles(const StepArgs& a, int i, int q, int chunk,
                                            unsigned char* smem, Sync& sync) {
  constexpr int NS = stages<HALVES>();
  const int tid = threadIdx.x;
  if (tid < NS) {
    tma::mbar_init(tma::smem_addr(&sync.full[tid]), 1);
    sync.left[tid] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const long long n = *a.step;
  const int tiles = a.n_orb_pad / kOrbitTile;
  // lane t looks at tile 16 i + t: is its block due in this chunk, and not yet formed
  const int lane = tid & 31, Tt = i * kAhead + lane;
  bool due = false;
  if (lane < kAhead && Tt < tiles) {
    const long long base = block_base(n, Tt);
    due = 1 + chunk * a.ahead_lc <= last_lag(a, base, Tt) &&
          a.stamp[((long long)chunk * tiles + Tt) * kSub + q] != block_mark(a, base);
  }
  unsigned todo = __ballot_sync(0xffffffffu, due);
  if (gridDim.z > 1) todo &= 1u << blockIdx.z;   // spread: one CTA per tile of the group
  __syncthreads();   // barriers ready; every warp has read the stamps
  unsigned g = 0;    // stages of the items before this one
  for (; todo; todo &= todo - 1) {
    if (tid == 0) sync.it.set(a, i * kAhead + __ffs(todo) - 1, q, chunk, n);
    __syncthreads();
    if (tid == 0) {
      const int first = min(NS, 2 * sync.it.nblk);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      sync.requested = g + first;
      for (int j = 0; j < first; ++j) request_stage<S, HALVES>(a, j, g + j, smem, sync);
    }
    const bool ok = sum_item<S, HALVES>(a, q, smem, sync, g);
    if (!__syncthreads_and(ok)) {
      if (tid == 0) {
        atomicExch(a.err, 1);
        // land the copies in flight before the CTA's shared memory is released
        for (unsigned s = sync.requested < NS ? 0 : sync.requested - NS; s < sync.requested; ++s)
          tma::mbar_wait(tma::smem_addr(&sync.full[s % NS]), (s / NS) & 1u, &tma::kNoError);
      }
      return;
    }
    g += 2 * sync.it.nblk;
    if (tid == 0)
      a.stamp[((long long)chunk * tiles + sync.it.T) * kSub + q] = block_mark(a, sync.it.base);
    __syncthreads();   // the item is read before the next replaces it
  }
}

// The weights of every (record half, lag) as the stages read them: [32 records][lag]
// [record (x 2 halves)][4], zero past the cutoff.  They depend on the handle alone:
// interpolated once, in double and rounded once (interpolating them in the summing
// kernel took its FP32 pipe and a warp's latency: 1.21 ms for 1024^2 x 4096 with a
// warp set aside for it, 1.23 with all, against 1.16).
template <bool HALVES>
__global__ void __launch_bounds__(256) ahead_weights_kernel(const StepArgs a, float4* __restrict__ out) {
  constexpr int ROWS = (HALVES ? 2 : 1) * kRec;
  const long long lags = ahead_weight_lags(a.n_cut);
  const long long i = blockIdx.x * 256ll + threadIdx.x;
  if (i >= (long long)a.n_orb_pad / kRec * lags * ROWS) return;
  const int m = (int)(i / ROWS % lags);
  const long long rec0 = i / ROWS / lags * kRec;
  const long long x = HALVES ? 2 * rec0 + i % ROWS : 2 * (rec0 + i % ROWS);
  double w[4] = {0.0, 0.0, 0.0, 0.0};
  if (m < a.n_cut) {
    const unsigned long long us = a.ustep[x];    // dT / h in 32.32 fixed point
    lag_weights(reinterpret_cast<const Double4*>(a.table64), (unsigned long long)m * us,
                (double)us * (a.table_h * (1.0 / 4294967296.0)), w);
  }
  out[i] = make_float4((float)w[0], (float)w[1], (float)w[2], (float)w[3]);
}

template <class S, bool HALVES>
__global__ void __launch_bounds__(kThreads, 1) ahead_kernel(const __grid_constant__ StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) Sync sync;
  ahead_tiles<S, HALVES>(a, blockIdx.x / kSub, blockIdx.x % kSub, blockIdx.y, smem, sync);
}

// The same over the members of a batch: CTA item_prefix[s] + ... belongs to member s,
// 4 sub-tiles of each group of 16 tiles, chunk-major.  The weights of whole and half
// records are laid out differently: a batch that holds both is launched once for each,
// and the CTAs of the other members return at once.
template <class S, bool HALVES>
__global__ void __launch_bounds__(kThreads, 1)
ahead_batch_kernel(const StepArgs* __restrict__ args, const int* __restrict__ item_prefix, int nb) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) Sync sync;
  __shared__ StepArgs s_args;
  __shared__ int s_local;
  if (threadIdx.x == 0) {
    int s = 0;
    while (s + 1 < nb && item_prefix[s + 1] <= (int)blockIdx.x) ++s;
    s_args = args[s];
    s_local = blockIdx.x - item_prefix[s];
  }
  __syncthreads();
  if ((s_args.halves != 0) != HALVES) return;
  const int per_chunk = ahead_ctas(s_args.n_orb_pad);
  const int r = s_local % per_chunk;
  ahead_tiles<S, HALVES>(s_args, r / kSub, r % kSub, s_local / per_chunk, smem, sync);
}

// A step's sums of one member (one thread): the current spectra rotated into the
// (xi, 2, perp) frame and stored in the ring, the chunks' block sums in chunk
// order, the lags 0 .. n - base inside the block, then the modal operator (the
// instantaneous coupling, -side mu |k|, rotation back).  Virtual members of one
// Nyquist bin are neighbouring lanes; the first adds them up and writes the bin.
template <class S>
__device__ __forceinline__ void near_member(const StepArgs& a, int T, int x) {
  using IO = MemberIO<S>;
  const int rec = T * kOrbitTile + (x >> 2);
  const long long mi = (long long)rec * kMembers + (x & 3);
  const int hx = 2 * rec + ((x >> 1) & 1);                // the member's half
  const long long n = *a.step;
  const long long base = block_base(n, T);
  const int s = (int)(n - base);
  const int sn = (int)(n % a.n_cut);
  const long long comp_stride = (long long)a.n_orb_pad * kMembers;

  const int b = a.bin[mi];
  const float2 e = reinterpret_cast<const float2*>(a.dir)[mi];
  float2 D[3];
  rotate_member(a, (int)mi, D);
  float2 R[3];   // as stored
#pragma unroll
  for (int c = 0; c < 3; ++c)
    R[c] = IO::store(a.hist, ((long long)sn * 3 + c) * comp_stride + mi, a.slot_stride, D[c]);

  float acc[kFields], cmp[kFields];
#pragma unroll
  for (int k = 0; k < kFields; ++k) acc[k] = cmp[k] = 0.f;
  auto fold = [&](int k, float v) {
    const float yy = v - cmp[k];
    const float t = acc[k] + yy;
    cmp[k] = (t - acc[k]) - yy;
    acc[k] = t;
  };
  auto lag = [&](const float w[4], const float2 (&d)[3]) {
    kadd<1>(acc[0], cmp[0], w[0], d[0].x); kadd<1>(acc[1], cmp[1], w[0], d[0].y);
    kadd<1>(acc[2], cmp[2], w[2], d[2].x); kadd<1>(acc[3], cmp[3], w[2], d[2].y);
    kadd<1>(acc[4], cmp[4], w[1], d[1].x); kadd<1>(acc[5], cmp[5], w[1], d[1].y);
    kadd<1>(acc[6], cmp[6], w[3], d[1].x); kadd<1>(acc[7], cmp[7], w[3], d[1].y);
    kadd<1>(acc[8], cmp[8], w[3], d[0].x); kadd<1>(acc[9], cmp[9], w[3], d[0].y);
  };
  // (issuing the next four lags' loads ahead of these took 56.6 instead of 52.3 us at
  // 1024^2, 123 registers against 92, and changed nothing below 512^2)
  // the chunks' block sums
  const int m_far = last_lag(a, base, T);
  const int nch = m_far > 0 ? (m_far + a.ahead_lc - 1) / a.ahead_lc : 0;
  const long long chunk_stride = comp_stride * kAhead * kFields;
  const float* P = a.ahead + (((long long)T * kAhead + s) * kFields) * (kOrbitTile * kMembers) + x;
  for (int ch = 0; ch < nch; ++ch) {
    float v[kFields];
#pragma unroll
    for (int k = 0; k < kFields; ++k) v[k] = __ldcs(P + ch * chunk_stride + k * (kOrbitTile * kMembers));
#pragma unroll
    for (int k = 0; k < kFields; ++k) fold(k, v[k]);
  }
  // lags inside the block, 4 in flight with their weights: those of the block sums,
  // rounded once from double (interpolating them in float from the table gave up to
  // 1.6 % more error and 1.3-2 us more a step up to 512^2, the same above)
  int M = min((int)(base < 0 ? n : n - base), a.n_cut - 1);
  if (a.tile_lmax) M = min(M, a.tile_lmax[T] - 1);
  const int lo = a.lmax ? a.lmax[hx] : 0x7fffffff;
  const int rows = kRec << a.halves;
  const float4* wrow = reinterpret_cast<const float4*>(a.wts32) +
                       (long long)(rec / kRec) * ahead_weight_lags(a.n_cut) * rows +
                       (a.halves ? hx % (2 * kRec) : rec % kRec);
  {
    const float4 q = __ldg(wrow);
    const float w[4] = {0.5f * q.x, 0.5f * q.y, 0.5f * q.z, 0.5f * q.w};
    lag(w, R);
  }
  for (int m = 1; m <= M; m += 4) {
    float2 d[4][3];
    float4 w4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (m + i <= M) {
        w4[i] = __ldg(wrow + (long long)(m + i) * rows);
        int slot = sn - (m + i);
        if (slot < 0) slot += a.n_cut;
#pragma unroll
        for (int c = 0; c < 3; ++c)
          d[i][c] = IO::load(a.hist, ((long long)slot * 3 + c) * comp_stride + mi, a.slot_stride);
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (m + i <= M) {
        const bool in = m + i < lo;
        const float w[4] = {in ? w4[i].x : 0.f, in ? w4[i].y : 0.f, in ? w4[i].z : 0.f, in ? w4[i].w : 0.f};
        lag(w, d[i]);
      }
  }

  // the modal operator
  float v[kFields];
#pragma unroll
  for (int k = 0; k < kFields; ++k) v[k] = acc[k] - cmp[k];
  const float muq = reinterpret_cast<const float*>(a.muq)[hx];
  const float sd = (float)a.side, inst = (float)(2.0 - a.eta);
  const float bxr = inst * D[1].x + v[6], bxi = inst * D[1].y + v[7];
  const float fxr = muq * (-sd * v[0] - bxi), fxi = muq * (-sd * v[1] + bxr);
  const float fpr = -sd * muq * v[2], fpi = -sd * muq * v[3];
  const float b2r = inst * D[0].x + v[8], b2i = inst * D[0].y + v[9];
  const float wsc = a.wout[mi] * (float)a.inv_n;
  float F[6];
  F[0] = wsc * (e.x * fxr - e.y * fpr);
  F[1] = wsc * (e.x * fxi - e.y * fpi);
  F[2] = wsc * (muq * (b2i - sd * v[4]));
  F[3] = wsc * (muq * (-b2r - sd * v[5]));
  F[4] = wsc * (e.y * fxr + e.x * fpr);
  F[5] = wsc * (e.y * fxi + e.x * fpi);
  const int g = x & 3;
  const int bp = __shfl_up_sync(0xffffffffu, b, 1, kMembers);
  const bool first = b >= 0 && !(g > 0 && bp == b);
  float G[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) G[k] = F[k];
#pragma unroll
  for (int d = 1; d < kMembers; ++d) {
    const int bd = __shfl_down_sync(0xffffffffu, b, d, kMembers);
    const bool take = g + d < kMembers && bd == b;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float z = __shfl_down_sync(0xffffffffu, F[k], d, kMembers);
      if (take) G[k] += z;
    }
  }
  if (first) {
    float2* fh = reinterpret_cast<float2*>(a.fhat);
    fh[b] = make_float2(G[0], G[1]);
    fh[a.nbins + b] = make_float2(G[2], G[3]);
    fh[2 * (long long)a.nbins + b] = make_float2(G[4], G[5]);
  }
}

constexpr int kNearThreads = 128, kNearSub = kOrbitTile * kMembers / kNearThreads;

template <class S>
__global__ void __launch_bounds__(kNearThreads) near_kernel(const StepArgs a) {
  near_member<S>(a, blockIdx.x / kNearSub, (blockIdx.x % kNearSub) * kNearThreads + threadIdx.x);
}

template <class S>
__global__ void __launch_bounds__(kNearThreads)
near_batch_kernel(const StepArgs* __restrict__ args, const int* __restrict__ tile_prefix, int nb) {
  const int t = blockIdx.x / kNearSub;
  int s = 0;
  while (s + 1 < nb && tile_prefix[s + 1] <= t) ++s;
  const StepArgs a = args[s];
  near_member<S>(a, t - tile_prefix[s], (blockIdx.x % kNearSub) * kNearThreads + threadIdx.x);
}

template <class S, bool HALVES>
cudaError_t prepare() {
  constexpr int bytes = smem_bytes<S, HALVES>();
  const cudaError_t e = cudaFuncSetAttribute(ahead_kernel<S, HALVES>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(ahead_batch_kernel<S, HALVES>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <class S, bool HALVES>
cudaError_t launch_sums(const StepArgs& a, cudaStream_t st, const BatchLaunch* batch) {
  constexpr int bytes = smem_bytes<S, HALVES>();
  if (batch) {
    ahead_batch_kernel<S, HALVES><<<dim3(batch->items, 1, a.spread ? kAhead : 1), kThreads, bytes, st>>>(
        batch->args, batch->item_prefix, batch->nb);
  } else {
    const dim3 grid(ahead_ctas(a.n_orb_pad), a.ahead_chunks, a.spread ? kAhead : 1);
    ahead_kernel<S, HALVES><<<grid, kThreads, bytes, st>>>(a);
  }
  return cudaGetLastError();
}

template <class S>
cudaError_t launch_near(const StepArgs& a, cudaStream_t st, const BatchLaunch* batch, int tiles) {
  if (batch)
    near_batch_kernel<S><<<tiles * kNearSub, kNearThreads, 0, st>>>(batch->args, batch->tile_prefix,
                                                                   batch->nb);
  else
    near_kernel<S><<<a.n_orb_pad / kOrbitTile * kNearSub, kNearThreads, 0, st>>>(a);
  return cudaGetLastError();
}

template <bool HALVES>
cudaError_t launch_weights(const StepArgs& a, cudaStream_t st) {
  const long long total = (long long)ahead_weight_bytes(a.n_orb_pad, a.n_cut, HALVES) / 16;
  ahead_weights_kernel<HALVES><<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
      a, reinterpret_cast<float4*>(const_cast<unsigned char*>(a.wts32)));
  return cudaGetLastError();
}

// One precision's entry: stage 0 sets the kernels' attributes, 1 launches the
// block sums, 2 the step's own sums and the assembly (over `tiles` tiles of a
// batch), 3 fills the handle's weights.
template <class S>
cudaError_t run_stage(const StepArgs& a, int stage, bool halves, cudaStream_t st,
                      const BatchLaunch* batch, int tiles) {
  switch (stage) {
    case 0: return halves ? prepare<S, true>() : prepare<S, false>();
    case 1: {
      const bool whole = batch ? batch->whole : !halves;
      cudaError_t e = whole ? launch_sums<S, false>(a, st, batch) : cudaSuccess;
      if (e == cudaSuccess && halves) e = launch_sums<S, true>(a, st, batch);
      return e;
    }
    case 3: return halves ? launch_weights<true>(a, st) : launch_weights<false>(a, st);
    case 2: return launch_near<S>(a, st, batch, tiles);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ahead
}  // namespace sbim
