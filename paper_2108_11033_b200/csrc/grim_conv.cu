// Tensor-core convolution for bf16 handles (Section 3.1: a convolution is a GEMM whose right-hand side is the expanded
// input; Section 4.5: that matrix is never produced in memory).
//
//   out[pixel, channel] = sum over (tap, input channel) of in[pixel shifted by tap, input channel] * W[channel, tap, input channel]
//
// Two launches.  conv_nhwc_kernel turns the NCHW input channel-last in a scratch of the handle (one pass, channels padded
// to a multiple of 8).  conv_tc_kernel then is a plain pipeline: TMA fetches the tile of input pixels of a tap straight
// from the channel-last copy (im2col mode: the copy engine walks rows and images, applies stride and padding), TMA fetches
// the tile of the expanded weights, one thread issues the multiplies, sixteen warps store the results (eight where others
// gather).  Pixels are the rows of the multiply, so a lane of the epilogue holds one pixel and a warp's store of one channel
// is contiguous in NCHW.
// Convolutions whose whole K fits one tile of 64 (few input channels: the first layer of a network) skip the
// channel-last copy: warps gather the tile of pixels from the NCHW input.
//
// The weights are expanded (zeros in place) once, when the matrix is packed: a convolution's matrix is small (4.7 MB for
// 512 x 512 x 3 x 3) and read from L2 by every pixel tile, so expanding packed records per tile, as the matrix kernels
// do, would only cost shared-memory bandwidth, which with the tensor core is what bounds the loop.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "grim_device.cuh"
#include "grim_internal.h"

namespace grim {
namespace {

using namespace ptx;

// ------------------------------------------------------------------------------------------ NCHW -> channel-last
// A thread block turns a 64-channel x 64-pixel tile around in shared memory.  Row pitch 65 elements: the eight lanes that
// read eight channels of one pixel then fall into different banks (8 * 65 * 2 bytes = 4 banks apart).
constexpr int kTrPitch = 65;
__global__ void __launch_bounds__(256) conv_nhwc_kernel(const unsigned short* __restrict__ in, unsigned short* __restrict__ out, int C, int Cp,
                                                        int hw, int vec) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ unsigned short t[64 * kTrPitch];
  const int p0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
  const int64_t img = blockIdx.z;
  in += img * C * hw;
  out += img * hw * Cp;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (vec) {  // planes of a multiple of 8 pixels: 16-byte loads
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int v = threadIdx.x + i * 256, c = v >> 3, p = (v & 7) * 8;
      uint4 u = make_uint4(0u, 0u, 0u, 0u);
      if (c0 + c < C && p0 + p < hw) u = __ldg(reinterpret_cast<const uint4*>(in + (int64_t)(c0 + c) * hw + p0 + p));
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        t[c * kTrPitch + p + 2 * e] = (unsigned short)w[e];
        t[c * kTrPitch + p + 2 * e + 1] = (unsigned short)(w[e] >> 16);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int v = threadIdx.x + i * 256, c = v >> 6, p = v & 63;
      t[c * kTrPitch + p] = (c0 + c < C && p0 + p < hw) ? __ldg(in + (int64_t)(c0 + c) * hw + p0 + p) : (unsigned short)0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int v = threadIdx.x + i * 256, p = v >> 3, c = (v & 7) * 8;
    if (p0 + p >= hw || c0 + c >= Cp) continue;
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w[e] = t[(c + 2 * e) * kTrPitch + p] | ((uint32_t)t[(c + 2 * e + 1) * kTrPitch + p] << 16);
    *reinterpret_cast<uint4*>(out + (int64_t)(p0 + p) * Cp + c0 + c) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// ------------------------------------------------------------------------------------------ the multiply
constexpr int kPix = 128;          // pixels per thread block: the rows of its accumulator
constexpr int kK = 64;             // k per stage
constexpr int kABytes = kPix * kK * 2;
constexpr int kMaxStages = 8;
constexpr int kEpiWarps = 8;       // of an epilogue group: two per quarter of the tensor-memory lanes
// Epilogue groups take tiles in turn: with few K tiles to a tile, storing it takes as long as multiplying it.  (Gathering, the
// warps are needed to build tiles.)
__host__ __device__ constexpr int epi_groups(bool gather) { return gather ? 1 : 2; }
constexpr int kEpi0 = 4;           // warps 0 and 3: pixel copies, 1: tensor core, 2: weight copies, from kEpi0 on the epilogue
constexpr int kThreads = 32 * (kEpi0 + kEpiWarps * epi_groups(false));
constexpr int kGatherGroups = 4;   // gathering variant: groups of four warps that build tiles of pixels in turn
constexpr int kGather0 = kEpi0 + kEpiWarps * epi_groups(true);  // their first warp
constexpr int kGatherThreads = 32 * kGather0 + 128 * kGatherGroups;
constexpr int kHdrBytes = 4096;
constexpr int kBiasCap = 512;      // output channels whose biases are kept in shared memory

struct ConvParams {
  unsigned* status;
  int nkt, nstages, npt, nnt;        // K tiles, ring slots, pixel tiles, channel tiles
  int n_tile, n_stride, nacc;        // output channels per tile; tensor-memory columns between accumulators; 2 or 4 of them
  int resident;                      // the weights of all K tiles stay in shared memory (one tile of output channels)
  int c_end;                         // a multiple of g past the last channel
  int g, cblocks;                    // channels per copy of input pixels, copies per tap
  int M, KH, KW, stride, pad, OH, OW;
  int C, H, W, K;
  int ksplit, kt_per;                // > 1: a cluster of ksplit blocks shares a tile, each multiplies kt_per K tiles
  int64_t npix;                      // images * OH * OW
  unsigned spin_limit;
  const __nv_bfloat16* X;            // gathering variant: the NCHW input
  const float* bias;
  void* Y;
  int y_bf16, relu;
};

__device__ __forceinline__ uint64_t k_major_desc(uint32_t saddr, int row_bytes) {
  // K-major tile with rows of 128, 64 or 32 bytes in the swizzle of that width: eight rows are row_bytes * 8 apart
  const uint64_t layout = row_bytes == 128 ? 2ull : (row_bytes == 64 ? 4ull : 6ull);
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)((row_bytes * 8) >> 4) << 32) | (1ull << 46) | (layout << 61);
}

template <int CG>
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accumulate) {
  if (CG == 1)
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate) : "memory");
  else
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate) : "memory");
}
template <int CG>
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  if (CG == 1)
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
  else  // in both blocks of the pair
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}
// Tile loads whose bytes are counted on a barrier given as a shared::cluster address (the even block's; no multicast).
template <int CG>
__device__ __forceinline__ void load_im2col(uint32_t dst, const void* map, int c, int w, int h, int n, unsigned short ow, unsigned short oh, uint32_t bar) {
  if (CG == 1)
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(ow), "h"(oh) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(ow), "h"(oh) : "memory");
}
template <int CG>
__device__ __forceinline__ void load_rows(uint32_t dst, const void* map, int x, int y, uint32_t bar) {
  if (CG == 1)
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void put(float* y, float t) { *y = t; }
__device__ __forceinline__ void put(__nv_bfloat16* y, float t) { *y = __float2bfloat16_rn(t); }
// n channels of one pixel, planes of ohw elements
template <typename T>
__device__ __forceinline__ void store_channels(T* y, int64_t ohw, int n, const float (&t)[32]) {
  if (n == 32) {
#pragma unroll
    for (int i = 0; i < 32; ++i) put(y + i * ohw, t[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i < n) put(y + i * ohw, t[i]);
  }
}

// CG = 2: two thread blocks on neighbouring SMs share a tile of 256 pixels (128 each) and n_tile channels; each stages
// its own pixels and half of the weight rows, the even one issues the multiplies for both.  That halves the weight bytes
// an SM reads per flop.  CG = 1: one block, 128 pixels - smaller tiles for small outputs.
// A thread block (pair) walks tiles blockIdx, blockIdx + grid, ...; two accumulators, so that storing a tile overlaps
// the multiplies of the next.
// GATHER: the tiles of pixels are gathered from the NCHW input (K <= 64).  KPS: K tiles per stage.
template <int CG, bool GATHER, int KPS>
__global__ void __launch_bounds__(GATHER ? kGatherThreads : kThreads, 1) conv_tc_kernel(const __grid_constant__ CUtensorMap tm_in,
                                                                                       const __grid_constant__ CUtensorMap tm_w, const ConvParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);   // (even block) the tiles of a stage have landed, both blocks' bytes
  uint64_t* empty = full + kMaxStages;                  // the multiplies of a stage are done
  uint64_t* acc_full = empty + kMaxStages;              // [nacc] an accumulator is complete
  uint64_t* acc_empty = acc_full + 4;                   // [nacc] (even block) it has been read by all warps of its group
  uint64_t* w_full = acc_empty + 4;                     // resident weights have landed (even block: both blocks' bytes)
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + 384);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + 388);
  int2* s_taps = reinterpret_cast<int2*>(smem + 1024);  // gathering variant: [k] (offset in the input, tap bits)
  float* s_bias = reinterpret_cast<float*>(smem + 2048);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
  const int b_rows = p.n_tile / CG;
  const uint32_t b_tile = ((uint32_t)b_rows * (kK * 2) + 1023u) & ~1023u;
  const bool resident = p.resident != 0;
  uint8_t* wbase = smem + kHdrBytes;  // resident weights
  const int wtiles = (p.nkt + KPS - 1) / KPS * KPS;
  uint8_t* stages = wbase + (resident ? (uint32_t)wtiles * b_tile : 0u);
  const uint32_t kt_bytes = (uint32_t)kABytes + (resident ? 0u : b_tile);
  const uint32_t stage_bytes = kt_bytes * (uint32_t)KPS;
  const bool split = CG == 1 && !GATHER && p.ksplit > 1;
  const uint32_t part = split ? cluster_ctarank() : 0u;  // this block's share of K
  const int kt0 = split ? (int)part * p.kt_per : 0;
  const int ns = p.nstages, nkt = split ? min(p.kt_per, p.nkt - kt0) : p.nkt;
  const int per = split ? p.ksplit : CG;                 // blocks per tile
  const int units = p.npt * p.nnt, u0 = (int)blockIdx.x / per, ustep = (int)gridDim.x / per;
  const uint32_t tmem_cols = (uint32_t)(p.nacc * p.n_stride);
  const int stages_per_tile = (nkt + KPS - 1) / KPS;

  if (tid == 32) {
    if (!GATHER) asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_in) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_w) : "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      // the copying threads of the even block announce the bytes of their loads; gathering: four warps arrive
      mbar_init(full + s, (GATHER ? 4 : 1) + (resident ? 0 : 1));
      mbar_init(empty + s, 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(acc_full + i, 1);
      mbar_init(acc_empty + i, kEpiWarps * CG);
    }
    mbar_init(w_full, 1);
    *s_abort = 0;
    fence_mbar_init();
  }
  if (GATHER && tid >= 32 * kGather0 && tid < 32 * kGather0 + kK) {
    // k -> (channel, kh, kw); tap bits: kh in the low half, 16 + kw in the high half (none valid past the last k)
    const int k = tid - 32 * kGather0, khw = p.KH * p.KW;
    const int c = k / khw, rest = k - c * khw, kh = rest / p.KW, kw = rest - kh * p.KW;
    s_taps[k] = k < p.K ? make_int2((c * p.H + kh) * p.W + kw, (int)((1u << kh) | (1u << (16 + kw)))) : make_int2(0, -1);
  }
  if (warp == 1) {
    if (CG == 1) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (CG == 2) cluster_sync_all();  // both blocks' barriers exist before either signals the other
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *s_tmem;
  // whatever earlier launches in the stream wrote - the channel-last copy of the input, the input, the biases - is complete and
  // visible from here on; up to here only the packed matrix and this block's own shared memory were touched
  asm volatile("griddepcontrol.wait;" ::: "memory");

  bool failed = false;
  int fail_site = 0;
  if (warp == 2) {
    // ------------------------------------------------------------------ weight copies
    // (a thread of their own: a copy costs the thread that issues it about 100 ns, and small tiles are done in less)
    if (elect_one()) {
      uint32_t full0 = smem_u32(full);  // the even block's barriers, as seen from this block
      if (CG == 2) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(full0) : "r"(smem_u32(full)), "r"(0));
      const uint32_t st0 = smem_u32(stages) + kABytes, b_bytes = (uint32_t)b_rows * (kK * 2);
      if (resident) {
        uint32_t wf = smem_u32(w_full);
        if (CG == 2) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(wf) : "r"(smem_u32(w_full)), "r"(0));
        if (rank == 0) mbar_arrive_expect_tx(w_full, b_bytes * (uint32_t)(wtiles * CG));  // (tiles past the last are zeros)
        for (int kt = 0; kt < wtiles; ++kt) load_rows<CG>(smem_u32(wbase) + (uint32_t)kt * b_tile, &tm_w, kt * kK, (int)rank * b_rows, wf);
      }
      // ring position: slot, and the parity of its last emptying (a fresh barrier counts as emptied one round before)
      int slot = 0;
      unsigned par = 1;
      for (int u = u0; u < units && !failed && !resident; u += ustep) {
        const int row0 = (u % p.nnt) * p.n_tile + (int)rank * b_rows;
        for (int stg = 0; stg < stages_per_tile; ++stg) {
          if (!mbar_wait_tight<CG == 2>(empty + slot, par, p.spin_limit, s_abort, 20)) { failed = true, fail_site = 5; break; }
          if (rank == 0) mbar_arrive_expect_tx(full + slot, b_bytes * (uint32_t)(KPS * CG));
#pragma unroll
          for (int j = 0; j < KPS; ++j)
            load_rows<CG>(st0 + (uint32_t)slot * stage_bytes + (uint32_t)j * kt_bytes, &tm_w, (kt0 + stg * KPS + j) * kK, row0, full0 + (uint32_t)slot * 8u);
          slot = slot + 1 == ns ? 0 : slot + 1;
          par ^= slot == 0 ? 1u : 0u;
        }
      }
    }
  } else if (warp == 0 || warp == 3) {
    // ------------------------------------------------------------------ pixel copies: two threads take stages in turn
    if (!GATHER && elect_one()) {
      uint32_t full0 = smem_u32(full);
      if (CG == 2) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(full0) : "r"(smem_u32(full)), "r"(0));
      const int ohw = p.OH * p.OW;
      const int subs = kK / p.g;
      const uint32_t st0 = smem_u32(stages), sub_bytes = (uint32_t)(kPix * p.g * 2);
      const int cut = KPS * subs;    // copies per stage
      int slot = warp == 0 ? 0 : 1, skip = slot;  // this thread's first stage, and how many of the next tile's come before it
      unsigned par = 1;
      for (int u = u0; u < units && !failed; u += ustep) {
        const int px = ((u / p.nnt) * CG + (int)rank) * kPix;  // first pixel of this block
        const int img = px / ohw, rest = px - img * ohw;
        const int oh = rest / p.OW, ow = rest - oh * p.OW;
        const int w0 = ow * p.stride - p.pad, h0 = oh * p.stride - p.pad;
        const int sub = kt0 * subs + skip * cut, tap = sub / p.cblocks;
        int cb = sub - tap * p.cblocks, tap_h = tap / p.KW, tap_w = tap - tap_h * p.KW;
        auto advance = [&]() {  // the next copy's channels and kernel position
          const bool wc = cb + 1 == p.cblocks;
          cb = wc ? 0 : cb + 1;
          tap_w += wc ? 1 : 0;
          const bool ww = tap_w == p.KW;
          tap_w = ww ? 0 : tap_w;
          tap_h += ww ? 1 : 0;
        };
        int stg = skip;
        for (; stg < stages_per_tile; stg += 2) {
          if (!mbar_wait_tight<CG == 2>(empty + slot, par, p.spin_limit, s_abort, 20)) { failed = true, fail_site = 1; break; }
          const uint32_t st = st0 + (uint32_t)slot * stage_bytes, bar = full0 + (uint32_t)slot * 8u;
          if (rank == 0) mbar_arrive_expect_tx(full + slot, sub_bytes * (uint32_t)(cut * CG));
#pragma unroll
          for (int j = 0; j < KPS; ++j)
            for (int i = 0; i < subs; ++i) {
              // a stage is always filled: copies past the last kernel position take channels that do not exist (zeros)
              const bool past = tap_h >= p.KH;
              load_im2col<CG>(st + (uint32_t)j * kt_bytes + (uint32_t)i * sub_bytes, &tm_in, past ? p.c_end : cb * p.g, w0, h0, img,
                              (unsigned short)(past ? 0 : tap_w), (unsigned short)(past ? 0 : tap_h), bar);
              advance();
            }
          for (int i = 0; i < cut; ++i) advance();
          slot += 2;
          const bool wrap = slot >= ns;
          slot -= wrap ? ns : 0;
          par ^= wrap ? 1u : 0u;
        }
        skip = stg - stages_per_tile;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ tensor core
    if (rank == 0 && elect_one()) {
      // fp32 accumulate, bf16 x bf16, both operands K-major, M = 128 pixels per block, N = n_tile channels
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.n_tile >> 3) << 17) | ((uint32_t)((kPix * CG) >> 4) << 24);
      const int row_bytes = p.g * 2, sub_shift = p.g == 64 ? 2 : (p.g == 32 ? 1 : 0);  // 16-wide k steps per copy: 4, 2, 1
      const uint64_t ad0 = k_major_desc(smem_u32(stages), row_bytes), bd0 = k_major_desc(resident ? smem_u32(wbase) : smem_u32(stages) + kABytes, 128);
      uint32_t step[kK / 16];  // where the k steps of a K tile start in the tile of pixels, in 16-byte units
#pragma unroll
      for (int s = 0; s < kK / 16; ++s) {
        const int sub = s >> sub_shift, in_sub = s - (sub << sub_shift);
        step[s] = (uint32_t)(sub * (kPix * row_bytes) + in_sub * 32) >> 4;
      }
      int slot = 0, tile = 0;
      unsigned par = 0;
      if (resident && !mbar_wait<CG == 2>(w_full, 0, p.spin_limit << 2, s_abort, 0)) failed = true, fail_site = 7;
      const uint32_t stage16 = stage_bytes >> 4, kt16 = kt_bytes >> 4;
      const uint32_t bstep = resident ? b_tile >> 4 : kt16;  // resident weights have places of their own
      const unsigned limit = p.spin_limit << 2;
      const int nacc = p.nacc, n_stride = p.n_stride;
      for (int u = u0; u < units && !failed; u += ustep, ++tile) {
        const int acc = tile & (nacc - 1), use = tile / nacc;
        if (!mbar_wait_tight<CG == 2>(acc_empty + acc, (unsigned)(use + 1) & 1u, limit, s_abort)) { failed = true, fail_site = 2; break; }
        const uint32_t d = tmem_base + (uint32_t)(acc * n_stride);
        uint32_t more = 0u, wk = 0u;
        for (int stg = 0; stg < stages_per_tile; ++stg) {
          if (!mbar_wait_tight<CG == 2>(full + slot, par, limit, s_abort)) { failed = true, fail_site = 3; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t off = (uint32_t)slot * stage16;  // (the address field of a descriptor never carries: 227 KB < 2^18)
          const uint32_t boff = resident ? wk : off;
#pragma unroll
          for (int j = 0; j < KPS; ++j)
#pragma unroll
            for (int s = 0; s < kK / 16; ++s)
              mma_bf16<CG>(d, ad0 + (off + (uint32_t)j * kt16 + step[s]), bd0 + (boff + (uint32_t)j * bstep + 2u * s), idesc, j + s > 0 ? 1u : more);
          mma_commit<CG>(empty + slot);
          more = 1u;
          wk += KPS * bstep;
          slot = slot + 1 == ns ? 0 : slot + 1;
          par ^= slot == 0 ? 1u : 0u;
        }
        if (!failed) mma_commit<CG>(acc_full + acc);
      }
    }
  } else if (GATHER && warp >= kGather0) {
    // ------------------------------------------------------------------ gathering variant: a thread builds one pixel's row
    const int grp = (warp - kGather0) >> 2, bt = (tid - 32 * kGather0) & 127;
    const int pieces = (p.K + 7) >> 3;  // 16-byte pieces of a row that hold something
    const unsigned short* X = reinterpret_cast<const unsigned short*>(p.X);
    const int ohw = p.OH * p.OW;
    int it = grp;
    for (int u = u0 + grp * ustep; u < units; u += kGatherGroups * ustep, it += kGatherGroups) {
      const int slot = it % ns;
      if (it >= ns && !__all_sync(0xffffffffu, mbar_wait(empty + slot, (unsigned)((it / ns - 1) & 1), p.spin_limit, s_abort, 32))) { failed = true, fail_site = 6; break; }
      const int q = (u / p.nnt) * kPix + bt;
      const bool ok = q < (int)p.npix;
      const int img = ok ? q / ohw : 0, pix = ok ? q - img * ohw : 0;
      const int oh = pix / p.OW, ow = pix - oh * p.OW;
      const int h0 = oh * p.stride - p.pad, w0 = ow * p.stride - p.pad;
      uint32_t in = 0;  // bit kh: row inside; bit 16 + kw: column inside
      for (int t = 0; t < p.KH; ++t) in |= (uint32_t)(ok && h0 + t >= 0 && h0 + t < p.H) << t;
      for (int t = 0; t < p.KW; ++t) in |= (uint32_t)(w0 + t >= 0 && w0 + t < p.W) << (16 + t);
      const int64_t base = ((int64_t)img * p.C * p.H + h0) * p.W + w0;
      const uint32_t row = smem_u32(stages) + (uint32_t)slot * stage_bytes + (uint32_t)bt * 128u;
#pragma unroll 2
      for (int pc = 0; pc < 8; ++pc) {
        uint32_t v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0u;
        if (pc < pieces) {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            // (selected, not skipped: a branch per element costs more than the load)
            const int2 t = s_taps[pc * 8 + e];
            const bool inside = (in & (uint32_t)t.y) == (uint32_t)t.y;
            const uint32_t x = __ldg(X + (inside ? base + t.x : 0));
            v[e] = inside ? x : 0u;
          }
        }
        sts128(row + (((uint32_t)pc ^ ((uint32_t)bt & 7u)) << 4), v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(full + slot);
    }
  } else {
    // ------------------------------------------------------------------ epilogue: a lane holds one pixel
    const int quarter = warp & 3;  // the tensor-memory lanes this warp may read
    const int64_t ohw = (int64_t)p.OH * p.OW;
    if (p.bias && p.M <= kBiasCap) {
      constexpr int kEpiThreads = 32 * kEpiWarps * epi_groups(GATHER);
      for (int i = tid - 32 * kEpi0; i < kBiasCap; i += kEpiThreads) s_bias[i] = i < p.M ? __ldg(p.bias + i) : 0.f;
      named_barrier(1, kEpiThreads);
    }
    // the accumulator has been read by this warp: the multiplies of a later tile may overwrite it once all warps say so
    auto release = [&](int acc) {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        if (CG == 1 || rank == 0) mbar_arrive(acc_empty + acc);
        else mbar_arrive_remote(acc_empty + acc, 0);
      }
    };
    const int egrp = (warp - kEpi0) / kEpiWarps, ewarp = (warp - kEpi0) % kEpiWarps;
    int tile = egrp;
    for (int u = u0 + egrp * ustep; u < units; u += epi_groups(GATHER) * ustep, tile += epi_groups(GATHER)) {
      const int acc = tile & (p.nacc - 1);
      if (!__all_sync(0xffffffffu, mbar_wait<CG == 2>(acc_full + acc, (unsigned)(tile / p.nacc) & 1u, p.spin_limit << 2, s_abort, 32))) { failed = true, fail_site = 4; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (split) break;  // one tile per cluster; the shares meet below
      const int pt = u / p.nnt, nt = u - pt * p.nnt;
      const int64_t px = ((int64_t)pt * CG + rank) * kPix + quarter * 32 + lane;
      const bool ok = px < p.npix;
      const int64_t img = ok ? px / ohw : 0;
      const int ch0 = nt * p.n_tile;
      const int64_t base = (img * p.M + ch0) * ohw + (ok ? px - img * ohw : 0);
      const int nch = p.M - ch0 < p.n_tile ? p.M - ch0 : p.n_tile;
      // Two neighbouring pixels per store where planes have an even size (then pixels 2i and 2i + 1 share an image): lanes
      // exchange halves so that even lanes hold both pixels of one channel and odd lanes of the next.
      const bool pairs = p.y_bf16 && (ohw & 1) == 0 && (reinterpret_cast<uintptr_t>(p.Y) & 3) == 0;
      const int cb0 = (ewarp >> 2) * 32;  // the two warps of a quarter take 32 channels in turn
      for (int cb = cb0; cb < nch; cb += 64) {
        uint32_t v[32];
        tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * p.n_stride + cb), v);
        if (cb + 64 >= nch) release(acc);
        const int n = nch - cb < 32 ? nch - cb : 32;
        float t[32];
        if (p.bias && p.M <= kBiasCap) {
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            // (ranges of channels start at multiples of 16; what is read past the last one is not stored)
            const float4 bv = *reinterpret_cast<const float4*>(s_bias + ((ch0 + cb + i) & (kBiasCap - 1)));
            t[i] = __uint_as_float(v[i]) + bv.x;
            t[i + 1] = __uint_as_float(v[i + 1]) + bv.y;
            t[i + 2] = __uint_as_float(v[i + 2]) + bv.z;
            t[i + 3] = __uint_as_float(v[i + 3]) + bv.w;
          }
        } else if (p.bias) {
#pragma unroll
          for (int i = 0; i < 32; ++i) t[i] = __uint_as_float(v[i]) + (i < n ? __ldg(p.bias + ch0 + cb + i) : 0.f);
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) t[i] = __uint_as_float(v[i]);
        }
        if (pairs) {
          // rounded channel by channel pair, activation on pairs, then one exchange and one byte permutation per pair
          const uint32_t sel = (lane & 1) ? 0x3276u : 0x5410u;
          uint32_t w[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            __nv_bfloat162 h = __floats2bfloat162_rn(t[2 * i], t[2 * i + 1]);
            if (p.relu) h = __hmax2(h, __floats2bfloat162_rn(0.f, 0.f));
            const uint32_t own = *reinterpret_cast<const uint32_t*>(&h);
            w[i] = __byte_perm(own, __shfl_xor_sync(0xffffffffu, own, 1), sel);
          }
          if (ok) {
            __nv_bfloat16* y = static_cast<__nv_bfloat16*>(p.Y) + base - (lane & 1) + (cb + (lane & 1)) * ohw;
            if (n == 32) {
#pragma unroll
              for (int i = 0; i < 16; ++i, y += 2 * ohw) *reinterpret_cast<uint32_t*>(y) = w[i];
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i, y += 2 * ohw)
                if (2 * i + (lane & 1) < n) *reinterpret_cast<uint32_t*>(y) = w[i];
            }
          }
        } else {
          if (p.relu)
#pragma unroll
            for (int i = 0; i < 32; ++i) t[i] = fmaxf(t[i], 0.f);
          if (ok) {
            if (p.y_bf16) store_channels(static_cast<__nv_bfloat16*>(p.Y) + base + cb * ohw, ohw, n, t);
            else store_channels(static_cast<float*>(p.Y) + base + cb * ohw, ohw, n, t);
          }
        }
      }
      if (cb0 >= nch) release(acc);  // nothing of this tile for this warp
    }
  }

  if (__any_sync(0xffffffffu, failed)) {
    *s_abort = 1;
    if (fail_site) atomicOr(p.status, (unsigned)GRIM_ERR_TIMEOUT | (1u << (8 + fail_site)));
  }
  if (split) {
    // Every block owns n_tile / ksplit of the tile's channels: each sends its sums to their owners' shared memory (the
    // stages are free once all blocks have multiplied) and the owner adds them up.  [block][channel][pixel] floats.
    __syncwarp();
    cluster_sync_all();
    const int nc = p.n_tile / p.ksplit;
    const bool epi = warp >= kEpi0 && warp < kEpi0 + kEpiWarps;
    if (epi) {
      const int quarter = warp & 3;
      const uint32_t dst = smem_u32(stages) + ((uint32_t)part * (uint32_t)nc * kPix + (uint32_t)(quarter * 32 + lane)) * 4u;
      for (int cb = ((warp - kEpi0) >> 2) * 32; cb < p.n_tile; cb += 64) {
        uint32_t v[32];
        tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)cb, v);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int owner = (cb + i) / nc, c = cb + i - owner * nc;
          uint32_t at;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(dst + (uint32_t)c * (kPix * 4)), "r"(owner));
          asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(v[i]) : "memory");
        }
      }
    }
    __syncwarp();
    cluster_sync_all();
    if (epi) {
      const float* sums = reinterpret_cast<const float*>(stages);
      const int pt = u0 / p.nnt, nt = u0 - pt * p.nnt;
      const int t = tid - 32 * kEpi0, pl = t & (kPix - 1);
      const int64_t px = (int64_t)pt * kPix + pl, ohw = (int64_t)p.OH * p.OW;
      if (px < p.npix) {
        const int64_t img = px / ohw, pix = px - img * ohw;
        for (int c = t / kPix; c < nc; c += 32 * kEpiWarps / kPix) {
          const int ch = nt * p.n_tile + (int)part * nc + c;
          if (ch >= p.M) break;
          float sum = 0.f;
          for (int s = 0; s < p.ksplit; ++s) sum += sums[(s * nc + c) * kPix + pl];
          if (p.bias) sum += __ldg(p.bias + ch);
          if (p.relu) sum = fmaxf(sum, 0.f);
          const int64_t off = (img * p.M + ch) * ohw + pix;
          if (p.y_bf16) put(static_cast<__nv_bfloat16*>(p.Y) + off, sum);
          else put(static_cast<float*>(p.Y) + off, sum);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*s_abort) let_copies_land();
  if (CG == 2) cluster_sync_all();  // neither block leaves (or frees tensor memory) while the other may still use its memory
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (CG == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------------------------------ host side
// The driver's tensor-map encoders, looked up through the runtime so that the library does not link against the driver.
template <typename F>
F driver_entry(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  return reinterpret_cast<F>(p);
}
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
using EncodeIm2colFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const int*,
                                    const int*, cuuint32_t, cuuint32_t, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
  static const EncodeTiledFn fn = driver_entry<EncodeTiledFn>("cuTensorMapEncodeTiled");
  return fn;
}
EncodeIm2colFn encode_im2col_fn() {
  static const EncodeIm2colFn fn = driver_entry<EncodeIm2colFn>("cuTensorMapEncodeIm2col");
  return fn;
}

bool gathers(const grim_bcr* h) { return h->conv[kConvGather].d_w != nullptr; }
const ConvLayout* layout_for(const grim_bcr* h, const SpmmArgs& a) {
  if (gathers(h)) return a.KH <= 16 && a.KW <= 16 ? &h->conv[kConvGather] : nullptr;
  for (const ConvLayout& l : h->conv)
    if (l.d_w && l.taps == a.KH * a.KW && (int64_t)a.C * l.taps == h->K) return &l;
  return nullptr;
}
int64_t images_of(const SpmmArgs& a) { return a.ncols / ((int64_t)a.OH * a.OW); }
int padded_channels(int C) { return (C + 7) / 8 * 8; }
size_t nhwc_bytes(const SpmmArgs& a) { return (size_t)images_of(a) * a.H * a.W * padded_channels(a.C) * 2; }

struct ConvPlan {
  int cg, n_tile, nnt, npt, ksplit, kt_per, grid;
};
bool shape_plan(ConvPlan& pl, int nkt, int64_t npix, int64_t M, int sms) {
  pl.nnt = (int)((M + pl.n_tile - 1) / pl.n_tile);
  const int64_t npt = (npix + kPix * pl.cg - 1) / (kPix * pl.cg);
  if (npt * pl.nnt > (int64_t(1) << 30)) return false;
  pl.npt = (int)npt;
  pl.kt_per = (nkt + pl.ksplit - 1) / pl.ksplit;
  if (pl.ksplit > 1) pl.kt_per = (pl.kt_per + 1) / 2 * 2;  // whole stages
  if (pl.ksplit > 1) {
    // one tile per cluster, every block with something to multiply; the sums have to fit the stages
    if (pl.cg != 1 || (pl.ksplit - 1) * pl.kt_per >= nkt || pl.n_tile % 32 || pl.n_tile % pl.ksplit) return false;
    pl.grid = pl.npt * pl.nnt * pl.ksplit;
    return pl.n_tile * kPix * 4 <= 128 * 1024;
  }
  pl.grid = (int)std::min<int64_t>(npt * pl.nnt, sms / pl.cg) * pl.cg;
  return true;
}
// Tile shape: the candidate with the lowest estimated time, in ns.  A K tile costs the slowest of: the thread that issues a
// copy (140), its bytes at the rate at which L2 feeds an SM's shared memory (120 per ns; 17 - 21 TB/s were measured over the
// GPU), the multiplies (shared-memory reads of both operands at 128 bytes a cycle included).  A tile's store overlaps the next
// tile's multiplies, the last one's does not; tiles are counted in whole waves.  The split over K trades a shorter loop for an
// exchange of about 2 us and is only considered where one wave holds all parts.
ConvPlan plan_for(int nkt, int64_t npix, int64_t M, int sms, bool gather) {
  ConvPlan best{};
  double best_t = -1.0;
  for (int cg = gather ? 1 : 2; cg >= 1; --cg)
    for (int n = 256; n >= 16 * cg; n -= 16 * cg)
      for (int ks = 1; ks <= 8; ks *= 2) {
        if (n > ((M + 31) / 32) * 32 || (ks > 1 && gather)) continue;
        ConvPlan pl{cg, n, 0, 0, ks, 0, 0};
        if (!shape_plan(pl, nkt, npix, M, sms)) continue;
        const int64_t units = (int64_t)pl.npt * pl.nnt;
        if (ks > 1 && units * ks > (ks == 8 ? 112 : sms - 8)) continue;
        const double mma = cg == 1 ? 128.0 + n : std::max(128.0 + n / 2, 1.0 * n);  // cycles
        const double kt = std::max(std::max(140.0, (kABytes + (double)n / cg * kK * 2) / 120.0), mma / 1.8);
        const double epi = 250.0 + 6.0 * n;
        const double waves = ks > 1 ? 1.0 : (double)((units + sms / cg - 1) / (sms / cg));
        const double t = waves * std::max(pl.kt_per * kt, epi) + epi + (ks > 1 ? 2000.0 : 0.0) + (cg == 2 ? 1000.0 : 0.0);
        if (best_t < 0.0 || t < best_t) { best_t = t; best = pl; }
      }
  return best;
}

}  // namespace

// Tensor map of an fp32 matrix with contiguous rows (16-byte aligned, a multiple of four values apart).
bool matrix_map_f32(const void* X, int64_t cols, int64_t rows, int64_t ld, int box_cols, int box_rows, void* map) {
  if (!encode_tiled_fn()) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
  const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows}, estr[2] = {1, 1};
  return encode_tiled_fn()(static_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(X), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Channels per copy of input pixels for a convolution with `taps` kernel positions: as few K tiles as possible.
ConvLayout conv_layout_shape(int64_t K, int taps) {
  ConvLayout best;
  const int64_t C = K / taps;
  for (int g = 64; g >= 16; g /= 2) {
    const int64_t cblocks = (C + g - 1) / g, nkt = (taps * cblocks * g + kK - 1) / kK;
    if (best.taps == 0 || nkt < best.nkt) {
      best.taps = taps; best.g = g; best.cblocks = (int)cblocks; best.nkt = (int)nkt;
    }
  }
  return best;
}

size_t conv_scratch_bytes(const grim_bcr* h, int64_t max_ncols) {
  size_t need = 0;
  for (int i = 0; i < kConvGather && !gathers(h); ++i) {
    const ConvLayout& l = h->conv[i];
    if (!l.d_w) continue;
    const size_t same = (size_t)max_ncols * padded_channels((int)(h->K / l.taps)) * 2;  // stride 1: as many input pixels as outputs
    if (same > ((size_t)1 << 30)) continue;  // beyond what grim_bcr_reserve allocates: such calls run on other kernels
    need = std::max(need, std::max(same, std::min(4 * same, (size_t)512 << 20)));       // stride 2: four times as many
  }
  return need;
}

bool conv_tc_supported(const grim_bcr* h, const SpmmArgs& a) {
  if (h->device < 0 || !h->d_status || !a.conv || a.x_dtype != GRIM_BF16 || !layout_for(h, a)) return false;
  if (a.ncols > (int64_t(1) << 31) - 512 || (int64_t)a.C * a.H * a.W >= (int64_t(1) << 31) || !encode_tiled_fn()) return false;
  if (gathers(h)) return true;
  if (a.KH != a.KW || a.stride > 8 || a.pad > 127 || a.H > 65535 || a.W > 65535 || images_of(a) > 65535 || (a.C + 63) / 64 > 65535) return false;
  return h->d_tc_acc && h->scratch_bytes >= nhwc_bytes(a) && encode_im2col_fn();
}

grim_status_t launch_conv_tc(const grim_bcr* h, const SpmmArgs& a, cudaStream_t s) {
  if (!conv_tc_supported(h, a)) return GRIM_ERR_UNSUPPORTED;
  const ConvLayout& l = *layout_for(h, a);
  const bool gather = gathers(h);
  const int Cp = padded_channels(a.C), hw = a.H * a.W;
  const int64_t images = images_of(a);
  const ConvPlan pl = plan_for(l.nkt, a.ncols, h->M, sm_count(h->device), gather);
  if (pl.grid <= 0) return GRIM_ERR_UNSUPPORTED;

  ConvParams p;
  p.status = h->d_status;
  p.nkt = l.nkt; p.npt = pl.npt; p.nnt = pl.nnt; p.n_tile = pl.n_tile; p.ksplit = pl.ksplit; p.kt_per = pl.kt_per;
  p.nacc = pl.n_tile <= 128 ? 4 : 2;
  p.n_stride = pl.n_tile <= 32 ? 32 : (pl.n_tile <= 64 ? 64 : (pl.n_tile <= 128 ? 128 : 256));
  p.g = l.g; p.cblocks = l.cblocks;
  p.M = (int)h->M; p.KH = a.KH; p.KW = a.KW; p.stride = a.stride; p.pad = a.pad; p.OH = a.OH; p.OW = a.OW;
  p.c_end = (a.C + l.g - 1) / l.g * l.g;
  p.C = a.C; p.H = a.H; p.W = a.W; p.K = (int)h->K;
  p.npix = a.ncols; p.spin_limit = 1u << 20; p.X = static_cast<const __nv_bfloat16*>(a.X); p.bias = a.bias; p.Y = a.Y;
  p.y_bf16 = a.y_dtype == GRIM_BF16; p.relu = a.relu;
  const int b_rows = pl.n_tile / pl.cg;
  // Handing a stage over costs the threads on both sides more than the multiplies of a K tile of up to 128 channels take: two
  // K tiles then share a stage.
  const int kps = !gather && pl.n_tile <= 128 && pl.kt_per > 1 ? 2 : 1;
  const size_t b_tile = ((size_t)b_rows * kK * 2 + 1023) & ~size_t(1023);
  // a single tile of output channels with a short K: its weights are loaded once per thread block, not once per pixel tile
  const size_t weights = b_tile * ((l.nkt + kps - 1) / kps * kps);
  p.resident = pl.nnt == 1 && pl.ksplit == 1 && weights <= 80 * 1024;
  const size_t fixed = 1024 + kHdrBytes + (p.resident ? weights : 0), stage = (kABytes + (p.resident ? 0 : b_tile)) * kps;
  p.nstages = (int)std::min<size_t>(kMaxStages, (227 * 1024 - fixed) / stage);
  const size_t smem = fixed + p.nstages * stage;

  CUtensorMap tin, tw;
  memset(&tin, 0, sizeof(tin));
  memset(&tw, 0, sizeof(tw));
  if (!gather) {
    const cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)images};
    const cuuint64_t strides[3] = {(cuuint64_t)Cp * 2, (cuuint64_t)Cp * 2 * a.W, (cuuint64_t)Cp * 2 * hw};
    const int lower[2] = {-a.pad, -a.pad}, upper[2] = {a.pad - (a.KW - 1), a.pad - (a.KH - 1)};
    const cuuint32_t estr[4] = {1, (cuuint32_t)a.stride, (cuuint32_t)a.stride, 1};
    const CUtensorMapSwizzle sw = l.g == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (l.g == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    if (encode_im2col_fn()(&tin, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, h->d_tc_acc, dims, strides, lower, upper, (cuuint32_t)l.g, kPix, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return GRIM_ERR_CUDA;
  }
  const cuuint64_t wdims[2] = {(cuuint64_t)l.nkt * kK, (cuuint64_t)h->M};
  const cuuint64_t wstrides[1] = {(cuuint64_t)l.nkt * kK * 2};
  const cuuint32_t wbox[2] = {(cuuint32_t)kK, (cuuint32_t)b_rows}, westr[2] = {1, 1};
  if (encode_tiled_fn()(&tw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, l.d_w, wdims, wstrides, wbox, westr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return GRIM_ERR_CUDA;
  cudaError_t e = cudaSuccess;
  if (!gather) {
    e = launch_pdl(conv_nhwc_kernel, dim3((unsigned)((hw + 63) / 64), (unsigned)((Cp + 63) / 64), (unsigned)images), dim3(256), 0, s,
                   static_cast<const unsigned short*>(a.X), reinterpret_cast<unsigned short*>(h->d_tc_acc), a.C, Cp, hw,
                   (hw % 8 == 0 && reinterpret_cast<uintptr_t>(a.X) % 16 == 0) ? 1 : 0);
    count_launch();
    if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
  }
  auto kern = gather ? conv_tc_kernel<1, true, 1>
                     : (kps == 2 ? (pl.cg == 2 ? conv_tc_kernel<2, false, 2> : conv_tc_kernel<1, false, 2>)
                                 : (pl.cg == 2 ? conv_tc_kernel<2, false, 1> : conv_tc_kernel<1, false, 1>));
  if (ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem) != cudaSuccess) return GRIM_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)pl.grid);
  cfg.blockDim = dim3(gather ? kGatherThreads : kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)std::max(pl.cg, pl.ksplit);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pl.cg == 2 || pl.ksplit > 1 ? 2 : 1;
  e = cudaLaunchKernelEx(&cfg, kern, tin, tw, p);
  count_launch();
  if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
  return GRIM_OK;
}

}  // namespace grim
