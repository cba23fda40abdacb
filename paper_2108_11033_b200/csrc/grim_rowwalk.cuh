// One warp's share of Y = W * X on the row-chunk layout, read straight from global memory: the device code shared by
// the direct kernel (grim_direct.cu) and the batched GRU step (grim_gru.cu).
//
// A warp walks every `parts`-th block column of ONE row band and owns 32 * NC output columns; the partial sums of the
// band's rows stay in registers.  Per 8 kept columns it reads the activations of those columns (coalesced, from
// L1 / L2: every row of X that a block keeps is read once and reused by all kept rows, Section 4.4) and, one 16-byte
// load per lane, the chunk's weights, which go through a small per-warp buffer in shared memory so that a row's
// weights can be broadcast.  The loads of a chunk are issued while the chunk before it is multiplied.
//
// There is no block-wide pipeline to fill, nothing to wait for but one's own loads, and the code is small (rows are the
// only unrolled loop): that is what small and middle-sized products need, whose time is latency and not throughput.
#pragma once
#include <cuda_bf16.h>

#include <type_traits>

#include "grim_device.cuh"
#include "grim_internal.h"

namespace grim {

struct RowWalk {
  const RcHead* head;   // [schedule position][block column]
  const uint8_t* blob;
  int nbc, bw;
};
struct RowRange : RowWalk {  // only nbc block columns from j0 on, of `stride` that a band has
  int j0, stride;
};

constexpr int kWalkChunkFloats = 8 * 16 + 8;               // a chunk's weights (at most 16 rows x 8 columns) and a row of slack
constexpr int kWalkBufFloats = 2 * kWalkChunkFloats;       // per-warp weight buffer: two chunks

// What a lane needs to know about its output columns to read activations of X(k, q) = X[k * x_sk + q * x_sq], or of the
// expanded input of a convolution (Section 4.5: never produced in memory).
template <int NC, int XV>
struct WalkCols {
  const void* ptr[NC / XV];  // X at (k = 0, this lane's first column of vector v); clamped to a valid column
  unsigned valid[NC];        // convolution: bit kh | bit (16 + kw) set where the tap is inside
};

__device__ __forceinline__ void walk_ffma2(unsigned long long& acc, unsigned long long w2, unsigned long long x2) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(w2), "l"(x2));
}
__device__ __forceinline__ unsigned long long walk_pair(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}

// Column (relative to the tile's first) of a lane's c-th output.
template <int XV>
__device__ __forceinline__ int walk_col(int c, int lane) { return (c / XV) * 32 * XV + lane * XV + c % XV; }

template <int NC, int XV, typename XT, int CONV>
__device__ __forceinline__ void walk_setup(const SpmmArgs& a, int64_t q0, int lane, WalkCols<NC, XV>& wc) {
  const XT* X = static_cast<const XT*>(a.X);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    int64_t q = q0 + walk_col<XV>(c, lane);
    const bool ok = q < a.ncols;
    if (!ok) q = 0;
    if (CONV) {
      const int64_t ohw = (int64_t)a.OH * a.OW;
      const int64_t img = q / ohw;
      const int pix = (int)(q - img * ohw);
      const int oh = pix / a.OW, ow = pix - oh * a.OW;
      const int ih0 = oh * a.stride - a.pad, iw0 = ow * a.stride - a.pad;
      unsigned m = 0;
      for (int t = 0; t < a.KH; ++t) m |= (unsigned)(ih0 + t >= 0 && ih0 + t < a.H) << t;
      for (int t = 0; t < a.KW; ++t) m |= (unsigned)(iw0 + t >= 0 && iw0 + t < a.W) << (16 + t);
      wc.valid[c] = ok ? m : 0u;
      wc.ptr[c / XV] = X + img * a.C * a.H * a.W + (int64_t)ih0 * a.W + iw0;  // (XV = 1) only dereferenced where a tap is inside
    } else {
      if (c % XV == 0) wc.ptr[c / XV] = X + q * a.x_sq;
    }
  }
}

// Accumulates block columns part, part + parts, ... of the band at schedule position pos into acc (pairs of the lane's
// outputs; NC = 1 uses acc1).  wbuf: this warp's kWalkBufFloats floats.  before_x() runs once, after the first records
// have been requested and before X is first read.  SKIP: padding columns of a chunk are not read and count as zero; otherwise
// they read the block's first kept column again and meet zero weights, which makes a NaN of an infinity there.  (For every
// product it would cost 3 to 4 % of the wider ones and of the GRU step.)
//
// One chunk is in flight ahead of the one that is multiplied.  (Two were measured: no gain, the copies between register
// sets cost what the latency gave - these kernels issue instructions most of the time.)
template <int BH, int NC, int XV, typename XT, int CONV, bool SKIP, typename Walk, typename BeforeX>
__device__ __forceinline__ void row_walk(const Walk& w, const SpmmArgs& a, int pos, int part, int parts, const WalkCols<NC, XV>& wc,
                                         float* wbuf, int lane, float (&acc1)[NC == 1 ? BH : 1],
                                         unsigned long long (&acc2)[NC == 1 ? 1 : BH][NC == 1 ? 1 : NC / 2], BeforeX before_x) {
  constexpr int NP = NC == 1 ? 1 : NC / 2;
  constexpr bool RANGE = std::is_same<Walk, RowRange>::value;
  int j0 = 0;
  const uint4* heads = reinterpret_cast<const uint4*>(w.head);
  if constexpr (RANGE) {
    j0 = w.j0;
    heads += (int64_t)pos * w.stride + j0;
  } else {
    heads += (int64_t)pos * w.nbc;
  }
  // a batch of up to 32 blocks: lane l holds the head of block column part + parts * (32 * batch + l)
  int jb = -1;
  unsigned todo = 0;  // lanes of the batch whose block has not been walked yet
  uint4 l_head = make_uint4(0, 0, 0, 0);
  const int nbatch = (w.nbc - part + 32 * parts - 1) / (32 * parts);

  // cursor: the chunk whose loads are issued next
  uint32_t rec = 0, c0 = 0, c1 = 0, rm = 0;
  int kr = 0, kc = 0, ch = 0, k0 = 0;
  auto next = [&]() -> bool {
    if (++ch * kRcChunk < kc) {
      const uint2 cc = __ldg(reinterpret_cast<const uint2*>(w.blob + (size_t)rec * 16 + 8) + ch);
      c0 = cc.x; c1 = cc.y;
      return true;
    }
    while (todo == 0) {
      if (++jb >= nbatch) { kc = 0; return false; }
      const int j = part + parts * (jb * 32 + lane);
      l_head = j < w.nbc ? __ldg(heads + j) : make_uint4(0u, 0u, 0u, 0u);
      todo = __ballot_sync(0xffffffffu, l_head.y != 0);
    }
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    rec = __shfl_sync(0xffffffffu, l_head.x, src);
    const uint32_t d = __shfl_sync(0xffffffffu, l_head.y, src);
    c0 = __shfl_sync(0xffffffffu, l_head.z, src);
    c1 = __shfl_sync(0xffffffffu, l_head.w, src);
    rm = rc_head_rows(d);
    kc = rc_head_kc(d);
    kr = __popc(rm);
    ch = 0;
    k0 = (j0 + part + parts * (jb * 32 + src)) * w.bw;
    return true;
  };

  // the chunk whose loads are under way
  float x[8][NC];
  float4 wv = make_float4(0.f, 0.f, 0.f, 0.f);
  const uint32_t ldb = (uint32_t)a.x_sk * (uint32_t)sizeof(XT);  // (the host checks that it fits)
  auto fetch_w = [&]() {
    const int nch = (kc + kRcChunk - 1) / kRcChunk;
    const float4* wp = reinterpret_cast<const float4*>(w.blob + (size_t)rec * 16 + ((8 + nch * kRcChunk + 15) & ~15)) + ch * kr * 2;
    if (lane < 2 * kr) wv = __ldg(wp + lane);
  };
  auto fetch_x = [&]() {
    int koff = 0;
    unsigned tap = 0;
    const int live = kc - ch * kRcChunk;  // columns of the chunk from here on are padding
    const bool half = live <= 4;          // nothing in the second half of the chunk
    if (CONV) {
      // lanes 0 .. 7 take the chunk's columns apart into (channel, kh, kw)
      const int k = k0 + (int)(((lane & 4 ? c1 : c0) >> (8 * (lane & 3))) & 0xFFu);
      const int khw = a.KH * a.KW;
      const int c = k / khw, rest = k - c * khw;
      const int kh = rest / a.KW, kw = rest - kh * a.KW;
      koff = (c * a.H + kh) * a.W + kw;
      tap = (1u << kh) | (1u << (16 + kw));
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (e == 4 && half) break;  // (uniform)
      if (CONV) {
        const int off = __shfl_sync(0xffffffffu, koff, e);
        const unsigned t = __shfl_sync(0xffffffffu, tap, e);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          float v = 0.f;
          if ((!SKIP || e < live) && (wc.valid[c] & t) == t) v = to_f32(static_cast<const XT*>(wc.ptr[c / XV])[off]);
          x[e][c] = v;
        }
      } else {
        const uint32_t k = (uint32_t)k0 + (((e < 4 ? c0 : c1) >> (8 * (e & 3))) & 0xFFu);
        if (SKIP && e >= live) {  // (uniform)
#pragma unroll
          for (int c = 0; c < NC; ++c) x[e][c] = 0.f;
          continue;
        }
#pragma unroll
        for (int v = 0; v < NC / XV; ++v) {
          const XT* src = reinterpret_cast<const XT*>(static_cast<const uint8_t*>(wc.ptr[v]) + (uint64_t)k * ldb);
          if (XV == 4 && sizeof(XT) == 4) {
            const float4 t = __ldg(reinterpret_cast<const float4*>(src));
            x[e][v * XV] = t.x; x[e][v * XV + 1 % XV] = t.y; x[e][v * XV + 2 % XV] = t.z; x[e][v * XV + 3 % XV] = t.w;
          } else if (XV == 2 && sizeof(XT) == 4) {
            const float2 t = __ldg(reinterpret_cast<const float2*>(src));
            x[e][v * XV] = t.x; x[e][v * XV + 1 % XV] = t.y;
          } else {
            x[e][v] = to_f32(src[0]);  // columns past the last one read column 0 and are never stored
          }
        }
      }
    }
  };

  bool more = next();
  if (more) fetch_w();
  before_x();
  if (more) fetch_x();
  int buf = 0;
  while (more) {
    float* wb = wbuf + buf * kWalkChunkFloats;
    if (lane < 2 * kr) reinterpret_cast<float4*>(wb)[lane] = wv;
    float xc[8][NC];
#pragma unroll
    for (int e = 0; e < 8; ++e)
#pragma unroll
      for (int c = 0; c < NC; ++c) xc[e][c] = x[e][c];
    const unsigned crm = rm;
    const bool ctwo = kc - ch * kRcChunk > 4;
    __syncwarp();  // the weights are there for every lane (the other buffer was read before the sync of the round before)
    more = next();
    if (more) { fetch_w(); fetch_x(); }
    // A row's weights are requested while the row before it is multiplied: rows sit behind branches (one warp-uniform
    // test each), so nothing else would overlap the loads' latency.  The read past the last row stays in the buffers.
    const float4* wr = reinterpret_cast<const float4*>(wb);
    float4 w0 = wr[0], w1 = ctwo ? wr[1] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < BH; ++r) {
      if ((crm >> r) & 1u) {
        const float we[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
        wr += 2;
        w0 = wr[0];
        if (ctwo) w1 = wr[1];
        if (NC == 1) {
          float& acc = acc1[NC == 1 ? r : 0];
#pragma unroll
          for (int e = 0; e < 4; ++e) acc = fmaf(we[e], xc[e][0], acc);
          if (ctwo) {
#pragma unroll
            for (int e = 4; e < 8; ++e) acc = fmaf(we[e], xc[e][0], acc);
          }
        } else {
          unsigned long long(&acc)[NP] = acc2[NC == 1 ? 0 : r];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const unsigned long long w2 = walk_pair(we[e], we[e]);
#pragma unroll
            for (int pr = 0; pr < NP; ++pr) walk_ffma2(acc[pr], w2, walk_pair(xc[e][2 * pr], xc[e][(2 * pr + 1) % NC]));
          }
          if (ctwo) {
#pragma unroll
            for (int e = 4; e < 8; ++e) {
              const unsigned long long w2 = walk_pair(we[e], we[e]);
#pragma unroll
              for (int pr = 0; pr < NP; ++pr) walk_ffma2(acc[pr], w2, walk_pair(xc[e][2 * pr], xc[e][(2 * pr + 1) % NC]));
            }
          }
        }
      }
    }
    buf ^= 1;
  }
}

// Value of output c of row r from the accumulators.
template <int BH, int NC>
__device__ __forceinline__ float walk_value(const float (&acc1)[NC == 1 ? BH : 1],
                                            const unsigned long long (&acc2)[NC == 1 ? 1 : BH][NC == 1 ? 1 : NC / 2], int r, int c) {
  if (NC == 1) return acc1[NC == 1 ? r : 0];
  const unsigned long long v = acc2[NC == 1 ? 0 : r][NC == 1 ? 0 : c / 2];
  return __uint_as_float((unsigned)((c & 1) ? v >> 32 : v));
}

}  // namespace grim
