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
// measured on GB300, 0.54 ms for 1024^2 x 4096 against 7.1 ms for the bytes).
//
// Blocks are aligned and staggered: tile T (128 records) starts its blocks at the
// steps with (n + T) mod 16 = 0, so every step renews 1/16 of the tiles and costs
// the same.  A tile's block is a function of n and T only, and every sum has a
// fixed order, so a step's result does not depend on when its sums were formed: a
// restored checkpoint, a rewound or repeated step and a replayed graph give the
// same bits as the run they continue.  Each (chunk, tile, 8 records) carries a stamp
// of the block its sums belong to and of the arguments' chunking and window; sums
// whose stamp is not the current one are formed again, all on the device, so that a
// captured graph renews them as a direct step does.  sbim_reset and sbim_load, which
// change the ring itself, mark every stamp invalid.
#pragma once

#include <type_traits>

#include "../../include/sbim.h"
#include "sbim_conv_tma.cuh"
#include "sbim_device.cuh"

namespace sbim {
namespace ahead {

using namespace dev;

// Records per CTA: 8 records x 4 members x 5 complex sums = 160 threads, one
// complex sum of one member per thread.  A thread keeps 16 outputs (running sum
// and compensation, 64 registers) and a window of 16 weights, each held twice so
// that one two-lane multiply-add takes (re, im) (32 registers).
constexpr int kRec = kAheadRec, kSums = 5, kThreads = kRec * kMembers * kSums;
constexpr int kSub = kOrbitTile / kRec;     // CTAs per 128-record tile
constexpr int kStages = 4;                  // 16-lag stages of history in shared memory
// one record's 16 weights of one kernel: 16 x 8 bytes, padded against bank conflicts
constexpr int kWRow = kAhead * 8 + 16;

template <class S> __host__ __device__ constexpr int seg() { return kRec * S::kRecBytes; }
template <class S> __host__ __device__ constexpr int stage_bytes() { return kAhead * 3 * S::kPlanes * seg<S>(); }
template <bool HALVES> __host__ __device__ constexpr int wbuf_bytes() { return (HALVES ? 2 : 1) * 4 * kRec * kWRow; }
template <class S, bool HALVES> __host__ __device__ constexpr int smem_bytes() {
  return kStages * stage_bytes<S>() + 2 * wbuf_bytes<HALVES>();
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

// One member's value: in a staged segment (8 records), in the ring, and as stored.
template <class S> struct MemberIO;
template <> struct MemberIO<StoreF32> {
  __device__ static float2 smem(const unsigned char* p, int lane) {
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
  __device__ static float2 smem(const unsigned char* p, int lane) {
    float2 d = unpack_bf16(*reinterpret_cast<const unsigned*>(p + lane * 4));
    if (LO) {
      const float2 l = unpack_bf16(*reinterpret_cast<const unsigned*>(p + kRec * 16 + lane * 4));
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
// Largest lag m of the block sums A[s] of tile T: the history before `base`, the
// cutoff, and the tile's truncation window.
__device__ __forceinline__ int last_lag(const StepArgs& a, long long base, int T) {
  int m = a.n_cut - 1;
  if (base < m) m = (int)(base < 0 ? 0 : base);
  if (a.tile_lmax) m = min(m, a.tile_lmax[T] - 1);
  return m;
}

// Block sums of records 8 q .. 8 q + 7 of tile T over one chunk of lags.  Stages
// of 16 lags arrive by bulk copies (3 components x 8 records each); the 16 weights
// per record of the block after next are interpolated while a block is summed.
// Per block of 16 lags and output the terms are chained by multiply-adds and every
// 32 lags folded into the running sum with one compensated addition.
// Returns false if a bounded wait gave up.
template <class S, bool HALVES>
__device__ __forceinline__ bool ahead_item(const StepArgs& a, int T, int q, int chunk, long long base,
                                           int m_end, unsigned char* smem, unsigned long long* full,
                                           unsigned& gstage) {
  constexpr int SEG = seg<S>(), STAGE = stage_bytes<S>(), WBUF = wbuf_bytes<HALVES>();
  using IO = MemberIO<S>;
  using u64 = unsigned long long;
  const int tid = threadIdx.x, lane = tid & 31;
  const int f = tid >> 5;                        // the sum: C11, C33, C22, C12a, C12b
  const int comp = f == 0 || f == 4 ? 0 : (f == 1 ? 2 : 1);
  const int kern = f == 0 ? 0 : (f == 1 ? 2 : (f == 2 ? 1 : 3));
  const int rec0 = T * kOrbitTile + q * kRec;
  const long long orb = a.n_orb_pad;
  const int m0 = 1 + chunk * a.ahead_lc;
  const int m1 = min(m0 + a.ahead_lc - 1, m_end);           // last lag of this chunk
  const int nblk = (m1 - m0 + kAhead) / kAhead;
  const int bs = (int)(base % a.n_cut);
  unsigned char* wsm = smem + kStages * STAGE;

  const unsigned char* hist = reinterpret_cast<const unsigned char*>(a.hist);
  const long long plane_bytes = a.slot_stride * S::kRecBytes;
  // stage b: lags m0 + 16 b .. +15 (clipped to m1), one copy per lag, component and
  // plane, issued by the lanes of warp 0
  auto issue = [&](int b) {
    const int buf = (int)((gstage + b) % kStages);
    const int mb = m0 + b * kAhead;
    const int copies = min(kAhead, m1 - mb + 1) * 3 * S::kPlanes;
    const unsigned bar = tma::smem_addr(&full[buf]);
    if (lane == 0) tma::mbar_expect_tx(bar, (unsigned)(copies * SEG));
    __syncwarp();
    for (int i = lane; i < copies; i += 32) {
      const int pl = i % S::kPlanes, lc = i / S::kPlanes;   // lc = lag * 3 + component
      int slot = bs - (mb + lc / 3);
      if (slot < 0) slot += a.n_cut;
      tma::bulk_g2s(tma::smem_addr(smem + buf * STAGE + i * SEG),
                    hist + pl * plane_bytes + (((long long)slot * 3 + lc % 3) * orb + rec0) * S::kRecBytes,
                    SEG, bar);
    }
  };
  if (f == 0)
    for (int b = 0; b < min(kStages - 1, nblk); ++b) issue(b);

  // the weights of block b: (record half, lag) pairs over the CTA's threads
  const float4* tab = reinterpret_cast<const float4*>(a.table);
  auto weights = [&](int b) {
    constexpr int PAIRS = (HALVES ? 2 : 1) * kRec * kAhead;
#pragma unroll
    for (int r = 0; r < (PAIRS + kThreads - 1) / kThreads; ++r) {
      const int i = tid + r * kThreads;
      if (i < PAIRS) {
        const int l = i % kAhead, rh = i / kAhead;          // rh: record (x 2 + half)
        const int x = HALVES ? 2 * rec0 + rh : 2 * (rec0 + rh);
        const int m = m0 + b * kAhead + l;
        float w[4] = {0.f, 0.f, 0.f, 0.f};
        if (m < a.n_cut && (!a.lmax || m < a.lmax[x]))
          lag_weights(tab, (u64)m * a.ustep[x], reinterpret_cast<const float*>(a.dT)[x], w);
        unsigned char* p = wsm + (b & 1) * WBUF + rh * kWRow + l * 8;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          *reinterpret_cast<float2*>(p + k * ((HALVES ? 2 : 1) * kRec * kWRow)) = make_float2(w[k], w[k]);
      }
    }
  };
  weights(0);
  weights(1);
  __syncthreads();
  const int row = HALVES ? 2 * (lane >> 2) + ((lane >> 1) & 1) : lane >> 2;
  const unsigned char* wrow = wsm + (kern * (HALVES ? 2 : 1) * kRec + row) * kWRow;

  u64 sum[kAhead], y[kAhead], w[kAhead];
#pragma unroll
  for (int s = 0; s < kAhead; ++s) sum[s] = y[s] = 0ull;    // (0.f, 0.f)
#pragma unroll
  for (int s = 0; s < kAhead; s += 2) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(wrow + s * 8);
    w[s] = v.x;
    w[s + 1] = v.y;
  }

  bool ok = true;
  int done = 0;
  for (int b = 0; b < nblk; ++b) {
    const unsigned gi = gstage + b;
    const bool landed = tma::mbar_wait(tma::smem_addr(&full[gi % kStages]), (gi / kStages) & 1u, a.err);
    // every thread has left block b - 1: its stage and its weights may be replaced,
    // and the weights of block b + 1 are complete
    if (!__syncthreads_and(landed)) {
      ok = false;
      break;
    }
    if (f == 0 && b + kStages - 1 < nblk) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(b + kStages - 1);
    }
    done = b + 1;
    const unsigned char* st = smem + (gi % kStages) * STAGE + comp * S::kPlanes * SEG;
    const unsigned char* wnext = wrow + ((b + 1) & 1) * WBUF;
    const int mb = m0 + b * kAhead;
    // At lag l output s takes weight l + s of the window; slot l is then replaced
    // by weight l of the next block.
    auto block = [&](auto tail) {
      constexpr bool TAIL = decltype(tail)::value;
      ulonglong2 nw;
#pragma unroll
      for (int l = 0; l < kAhead; ++l) {
        float2 d = IO::smem(st + l * 3 * S::kPlanes * SEG, lane);
        if (TAIL && mb + l > m1) d = make_float2(0.f, 0.f);
        if (l % 2 == 0) nw = *reinterpret_cast<const ulonglong2*>(wnext + l * 8);
        const u64 dd = pack2(d);
#pragma unroll
        for (int s = 0; s < kAhead; ++s) {
          // terms past the cutoff are left out, not multiplied by zero: a
          // non-finite value leaves the sums with its last lag
          const u64 ds = TAIL && mb + l + s >= a.n_cut ? 0ull : dd;
          y[s] = fma2r(w[(l + s) % kAhead], ds, y[s]);
        }
        w[l] = l % 2 == 0 ? nw.x : nw.y;
      }
    };
    if (mb + 2 * kAhead - 2 < a.n_cut && mb + kAhead - 1 <= m1)
      block(std::false_type{});
    else
      block(std::true_type{});
    if (b + 2 <= nblk) weights(b + 2);
    if ((b & 1) || b + 1 == nblk) {
#pragma unroll
      for (int s = 0; s < kAhead; ++s) {
        const u64 t = add2r(sum[s], y[s]);
        y[s] = sub2r(y[s], sub2r(t, sum[s]));      // minus the compensation
        sum[s] = t;
      }
    }
  }
  if (!ok) {
    if (tid == 0) atomicExch(a.err, 1);
    const int issued = min(nblk, done + kStages - 1);   // land what is in flight
    for (int s = done; s < issued; ++s) {
      const unsigned gs = gstage + s;
      tma::mbar_wait(tma::smem_addr(&full[gs % kStages]), (gs / kStages) & 1u, &tma::kNoError);
    }
    return false;
  }
  gstage += nblk;
  float* out = a.ahead + (((long long)chunk * (orb / kOrbitTile) + T) * kAhead * kFields + 2 * f) *
                             (kOrbitTile * kMembers) + q * (kRec * kMembers) + lane;
#pragma unroll
  for (int s = 0; s < kAhead; ++s) {
    const float2 r = unpack2(add2r(sum[s], y[s]));
    float* o = out + (long long)s * kFields * (kOrbitTile * kMembers);
    o[0] = r.x;
    o[kOrbitTile * kMembers] = r.y;
  }
  __syncthreads();   // the weight buffers are free for the next tile
  return true;
}

// The tiles 16 i .. 16 i + 15 of one update, records 8 q .. of each, one chunk of
// lags: in a running time loop one of the 16 starts a new block at every step.
template <class S, bool HALVES>
__device__ __forceinline__ void ahead_tiles(const StepArgs& a, int i, int q, int chunk,
                                            unsigned char* smem, unsigned long long* full) {
  if (threadIdx.x == 0) {
#pragma unroll
    for (int b = 0; b < kStages; ++b) tma::mbar_init(tma::smem_addr(&full[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const long long n = *a.step;
  const int tiles = a.n_orb_pad / kOrbitTile;
  unsigned gstage = 0;
  for (int T = i * kAhead; T < min(tiles, (i + 1) * kAhead); ++T) {
    const long long base = block_base(n, T);
    const int m_end = last_lag(a, base, T);
    if (1 + chunk * a.ahead_lc > m_end) continue;
    long long* stamp = a.stamp + ((long long)chunk * tiles + T) * kSub + q;
    const long long mark = base * 65536 + a.config_id;
    if (*stamp == mark) continue;
    if (!ahead_item<S, HALVES>(a, T, q, chunk, base, m_end, smem, full, gstage)) return;
    if (threadIdx.x == 0) *stamp = mark;
  }
}

template <class S, bool HALVES>
__global__ void __launch_bounds__(kThreads, 3) ahead_kernel(const StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long full[kStages];
  ahead_tiles<S, HALVES>(a, blockIdx.x / kSub, blockIdx.x % kSub, blockIdx.y, smem, full);
}

// The same over the members of a batch: CTA item_prefix[s] + ... belongs to member s,
// 16 sub-tiles of each group of 16 tiles, chunk-major.
template <class S, bool HALVES>
__global__ void __launch_bounds__(kThreads, 3)
ahead_batch_kernel(const StepArgs* __restrict__ args, const int* __restrict__ item_prefix, int nb) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long full[kStages];
  __shared__ StepArgs s_args;
  __shared__ int s_local;
  if (threadIdx.x == 0) {
    int s = 0;
    while (s + 1 < nb && item_prefix[s + 1] <= (int)blockIdx.x) ++s;
    s_args = args[s];
    s_local = blockIdx.x - item_prefix[s];
  }
  __syncthreads();
  const int per_chunk = ahead_ctas(s_args.n_orb_pad);
  const int r = s_local % per_chunk;
  ahead_tiles<S, HALVES>(s_args, r / kSub, r % kSub, s_local / per_chunk, smem, full);
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
  if (b >= 0) {
    const float2* uh = reinterpret_cast<const float2*>(a.uhat);
    const float2 u1 = uh[b], u2 = uh[a.nbins + b], u3 = uh[2 * (long long)a.nbins + b];
    D[0] = make_float2(e.x * u1.x + e.y * u3.x, e.x * u1.y + e.y * u3.y);
    D[1] = u2;
    D[2] = make_float2(-e.y * u1.x + e.x * u3.x, -e.y * u1.y + e.x * u3.y);
  } else {
    D[0] = D[1] = D[2] = make_float2(0.f, 0.f);
  }
  float2 R[3];   // as stored
#pragma unroll
  for (int c = 0; c < 3; ++c)
    R[c] = IO::store(a.hist, ((long long)sn * 3 + c) * comp_stride + mi, a.slot_stride, D[c]);

  const float4* tab = reinterpret_cast<const float4*>(a.table);
  const float dT = reinterpret_cast<const float*>(a.dT)[hx];
  const unsigned long long us = a.ustep[hx];
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
  // chunks of the block sums, two at a time in flight
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
  // lags inside the block, 4 in flight
  int M = min((int)(base < 0 ? n : n - base), a.n_cut - 1);
  if (a.tile_lmax) M = min(M, a.tile_lmax[T] - 1);
  const int lo = a.lmax ? a.lmax[hx] : 0x7fffffff;
  {
    float w[4];
    lag_weights(tab, 0ull, dT * 0.5f, w);
    lag(w, R);
  }
  for (int m = 1; m <= M; m += 4) {
    float2 d[4][3];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (m + i <= M) {
        int slot = sn - (m + i);
        if (slot < 0) slot += a.n_cut;
#pragma unroll
        for (int c = 0; c < 3; ++c)
          d[i][c] = IO::load(a.hist, ((long long)slot * 3 + c) * comp_stride + mi, a.slot_stride);
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (m + i <= M) {
        float w[4];
        lag_weights(tab, (unsigned long long)(m + i) * us, m + i < lo ? dT : 0.f, w);
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
    ahead_batch_kernel<S, HALVES><<<batch->items, kThreads, bytes, st>>>(batch->args, batch->item_prefix,
                                                                        batch->nb);
  } else {
    const dim3 grid(ahead_ctas(a.n_orb_pad), a.ahead_chunks);
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

// One precision's entry: stage 0 sets the kernels' attributes, 1 launches the
// block sums, 2 the step's own sums and the assembly (over `tiles` tiles of a batch).
template <class S>
cudaError_t run_stage(const StepArgs& a, int stage, bool halves, cudaStream_t st,
                      const BatchLaunch* batch, int tiles) {
  switch (stage) {
    case 0: return halves ? prepare<S, true>() : prepare<S, false>();
    case 1: return halves ? launch_sums<S, true>(a, st, batch) : launch_sums<S, false>(a, st, batch);
    case 2: return launch_near<S>(a, st, batch, tiles);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ahead
}  // namespace sbim
