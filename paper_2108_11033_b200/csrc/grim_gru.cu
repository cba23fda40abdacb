// GRU sequence inference built from the BCR matrix-vector product (Section 3.1: RNN layers are
// matrix-vector multiplications; Section 6.1: a 2-layer GRU is the RNN workload).
//
// Per layer: (1) the input-side products W_ih x_t for all T steps do not depend on the recurrence and
// are hoisted into one sparse GEMM with N = T (bias b_ih fused); (2) one persistent kernel walks the T
// dependent steps.  Every thread block owns some groups of bh hidden units and the three row bands
// (r, z, n gates) of W_hh that produce them; it copies those bands' packed chunks into shared memory
// once, so that W_hh is read from HBM once per sequence instead of once per step.  Per step the blocks
// multiply their bands with h_{t-1}, apply the gate non-linearities and exchange their slices of h_t.
//
// Exchange schemes:
//   gru_cluster_reg_kernel, gru_stack_kernel
//                         one cluster holds W_hh in registers; of a stack of two or three layers all run in one launch, a few
//                         steps behind each other.  Used whenever the layers fit.
//   gru_cluster_kernel    one thread-block cluster (up to 16 CTAs) holds all of W_hh; h_t is broadcast
//                         with distributed-shared-memory stores and the step ends with the hardware
//                         cluster barrier.  Used whenever the layer fits one cluster.
//   gru_recurrent_kernel  cooperative grid of up to 128 CTAs; h_t goes through L2 and the step ends with a
//                         grid-wide barrier in global memory whose wait is bounded (status word on expiry).
#include <cooperative_groups.h>

#include <algorithm>
#include <future>
#include <new>
#include <numeric>

#include "grim_device.cuh"
#include "grim_internal.h"
#include "grim_rowwalk.cuh"

namespace cg = cooperative_groups;
using namespace grim;

namespace {
constexpr int kMaxLocalBands = 48;
struct ModeCfg {
  int tpc = 1, ks = 1, threads = 0, ctas = 0, resident = 0;
  uint32_t max_chunks = 0, max_cw = 0, max_vals = 0;
  size_t smem = 0;
  bool ok = false;
};
}  // namespace

namespace { struct GruParams; struct GruStack; }

struct grim_gru {
  int L = 0;
  int64_t H = 0, max_T = 0;
  int bh = 0;
  std::vector<const grim_bcr*> Wih, Whh;
  std::vector<float*> d_bih, d_bhh;
  std::vector<uint32_t*> d_pos_of_band;     // schedule position of every band of W_hh
  std::vector<uint32_t*> d_pos_of_band_ih;  // ... of W_ih
  std::vector<float*> d_img_val;      // register images of the register-resident kernels (may be empty): W_hh of every layer, and where
                                      // the layers run in one launch W_hh from number stack_hh on, W_ih of layer l at stack_ih + l
  std::vector<uint32_t*> d_img_col;
  std::vector<float*> d_gi_saved;  // grim_gru_seq_static parks d_gi here while it points the pass at the static array
  std::vector<float*> d_gi;  // per layer: hoisted pre-activations, T x 3H (layers overlap in time, so each has its own)
  float* d_seq[2] = {nullptr, nullptr};
  // unit-major copies (feature x time, row stride = T rounded up to 4): the projections then read X row-major
  float* d_seqT[2] = {nullptr, nullptr};
  float* d_xT = nullptr;
  bool transposed_inputs = true;
  // layer pipelining: layer l runs on its own stream, a chunk of time steps behind layer l - 1
  std::vector<cudaStream_t> lstream;   // streams of layers 1 .. L-1 (layer 0 uses the caller's stream)
  std::vector<cudaStream_t> pstream;   // their input projections: chunk c + 1 is projected while the recurrence is on chunk c
  std::vector<cudaEvent_t> ev_proj;    // [layer][chunk]: the chunk's projection is there
  std::vector<cudaEvent_t> ev_chunk;   // [layer][chunk]: the layer's recurrence has produced the chunk
  cudaEvent_t ev_fork = nullptr;
  int max_chunks = 8;
  bool pipeline = true;
  int want_chunks = 0;  // 0: chosen from T
  unsigned* d_sync = nullptr;  // [0..L): barrier counters, [L]: status word
  ModeCfg grid, cluster;       // launch shapes of the shared-memory kernels
  ModeCfg regc;                // launch shape of the register-resident cluster kernel
  void (*reg_kern)(const GruParams) = nullptr;    // its compiled variant
  int stack_hh = 0, stack_ih = 0;
  ModeCfg stack;                                  // launch shape of the same variant for all layers in one launch
  void (*stack_kern)(const GruStack) = nullptr;
  int device = -1;
  cudaStream_t last_stream = nullptr;
  int dbg_skip_cta = -1;
  float* d_never = nullptr;  // (test hook) pre-activations that never arrive
  unsigned spin_limit = 1u << 22;
  bool force_grid = false;
  bool profile = false;
  std::vector<cudaEvent_t> ev;  // timing events, used in pairs: (before, after) each projection / recurrent launch
  std::vector<int> ev_kind;     // 0 / 1: before / after a projection, 2 / 3: before / after a recurrent kernel
  int ev_used = 0;
};

namespace {

struct GruParams {
  const uint32_t* band_ptr;
  const ChunkDesc* chunks;
  const uint32_t* colwords;
  const float* vals;
  const uint32_t* pos_of_band;
  const float* b_hh;
  const float* gi;   // T x 3H, b_ih already added
  const float* b_ih; // 3H or null: added to gi here
  const float* h0;   // H or null
  float* out;        // T x H
  float* outT;       // null, or the same values unit-major: outT[unit * ldT + t] (input of the next layer's projection)
  int64_t ldT;
  float* hT;         // H or null
  unsigned* bar;
  unsigned* status;
  int H, bh, T, tpc, ks, resident;
  uint32_t max_chunks, max_cw, max_vals;
  int skip_cta;
  unsigned spin_limit;
  // register image of the register-resident kernels: what every thread keeps for the whole sequence, laid out
  // so that the threads of a block read consecutive words ([cta][item][slot][row or column][thread])
  const float* img_val;
  const uint32_t* img_col;
};

// The stacked kernel: cluster c of a launch plays role[c], an even one the recurrence of layer c / 2, an odd one the
// projection of layer (c + 1) / 2.
constexpr int kMaxStack = 3;                    // layers in one launch
constexpr int kWithhold = -2;                   // (grim_gru_debug_barrier)
constexpr unsigned kNotYet = 0xFFFFFFFFu;       // what buffers between clusters are filled with: a NaN that no arithmetic produces
struct GruRole {
  const float* img_val;
  const uint32_t* img_col;
  const float* bias;         // recurrence: b_hh, projection: b_ih
  const float* in;           // recurrence: pre-activations, T x 3H; projection: outputs of the layer below, T x H
  float* out;                // recurrence: T x H; projection: T x 3H
  const float* h0;           // H or null
  float* hT;                 // H or null
  int waits;                 // another cluster writes `in` in the same launch: kNotYet where it has not yet
};
struct GruStack {
  GruRole role[2 * kMaxStack - 1];
  unsigned* status;
  int H, bh, T, tpc, ks;
  unsigned spin_limit;
};

__device__ __forceinline__ void gru_mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void gru_mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool gru_mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Stores v at the place of CTA-local shared address `local` in CTA `rank` of the cluster and counts its 4 bytes on
// that CTA's mbarrier at CTA-local address `bar_local`.
__device__ __forceinline__ void gru_st_async_f32(uint32_t local, uint32_t bar_local, uint32_t rank, float v) {
  uint32_t raddr, rbar;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(local), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(bar_local), "r"(rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(raddr), "f"(v), "r"(rbar) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Values that another thread block of the same launch polls for: the value itself says that it is there.
__device__ __forceinline__ void st_shared_value(float* p, float v) { asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory"); }
__device__ __forceinline__ float ld_shared_value(const float* p) {
  float v;
  asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_shared_values(const float* p) {  // each of the four on its own
  float4 v;
  asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_gpu_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ float sigmoidf_(float v) { return 1.f / (1.f + expf(-v)); }

// tanh without a branch: the recurrent step waits for it, and lanes on both sides of a threshold would take both paths in
// turn.  Below 0.5 the Taylor series about 0 (eight terms, remainder below 1e-8 of the result), above it
// 1 - 2 / (1 + e^(2|x|)).  Within 2.1 units in the last place.
__device__ __forceinline__ float tanh_both(float x) {
  const float ax = fabsf(x), x2 = x * x;
  float p = 6404582.f / 10854718875.f;
  p = fmaf(p, x2, -929569.f / 638512875.f);
  p = fmaf(p, x2, 21844.f / 6081075.f);
  p = fmaf(p, x2, -1382.f / 155925.f);
  p = fmaf(p, x2, 62.f / 2835.f);
  p = fmaf(p, x2, -17.f / 315.f);
  p = fmaf(p, x2, 2.f / 15.f);
  p = fmaf(p, x2, -1.f / 3.f);
  const float small = fmaf(x * x2, p, x);
  const float big = fmaf(__frcp_rn(1.f + expf(2.f * ax)), -2.f, 1.f);
  return ax < 0.5f ? small : copysignf(big, x);
}

// Per-CTA view of its bands' chunks: either the global arrays or copies in shared memory.
struct BandView {
  const ChunkDesc* ch;
  const uint32_t* cw;
  const float* vals;
  const uint32_t* cb;  // chunk range per local band (local band = group * 3 + gate)
  const uint32_t* ce;
};

// One-time set-up: locate the bands of CTA `cta` (tpc groups of bh hidden units x 3 gates) and, if they
// fit, copy their chunk descriptors / column words / values into shared memory.  `pool` is the dynamic
// shared memory left after the caller's own arrays.
__device__ BandView setup_bands(const GruParams& p, int cta, uint8_t* pool) {
  __shared__ uint32_t s_src_c[kMaxLocalBands], s_src_cw[kMaxLocalBands], s_src_v[kMaxLocalBands];
  __shared__ uint32_t s_dst_cw[kMaxLocalBands], s_dst_v[kMaxLocalBands], s_n_cw[kMaxLocalBands], s_n_v[kMaxLocalBands];
  __shared__ uint32_t s_cb[kMaxLocalBands], s_ce[kMaxLocalBands];
  const int tid = threadIdx.x;
  const int nb = 3 * p.tpc;
  const int nbands_gate = p.H / p.bh;
  ChunkDesc* s_ch = reinterpret_cast<ChunkDesc*>(pool);
  uint32_t* s_cw = reinterpret_cast<uint32_t*>(s_ch + p.max_chunks);
  float* s_val = reinterpret_cast<float*>(s_cw + p.max_cw);
  if (tid == 0) {
    uint32_t nc = 0, ncw = 0, nv = 0;
    for (int lb = 0; lb < nb; ++lb) {
      const int tri = cta * p.tpc + lb / 3;
      uint32_t cb = 0, ce = 0;
      if (tri < nbands_gate) {
        const uint32_t pos = p.pos_of_band[(lb % 3) * nbands_gate + tri];
        cb = p.band_ptr[pos];
        ce = p.band_ptr[pos + 1];
      }
      uint32_t n_cw = 0, n_v = 0;
      for (uint32_t c = cb; c < ce; ++c) {
        const uint32_t nk = p.chunks[c].ncols_kr;
        n_cw += 32;  // every chunk owns 32 column words
        n_v += (nk & 0xFFFFu) * (nk >> 16);
      }
      s_src_c[lb] = cb;
      s_src_cw[lb] = cb < ce ? p.chunks[cb].cw_off : 0;
      s_src_v[lb] = cb < ce ? p.chunks[cb].val_off : 0;
      s_dst_cw[lb] = ncw; s_dst_v[lb] = nv; s_n_cw[lb] = n_cw; s_n_v[lb] = n_v;
      if (p.resident) { s_cb[lb] = nc; s_ce[lb] = nc + (ce - cb); }
      else { s_cb[lb] = cb; s_ce[lb] = ce; }
      nc += ce - cb; ncw += n_cw; nv += n_v;
    }
  }
  __syncthreads();
  BandView v{p.chunks, p.colwords, p.vals, s_cb, s_ce};
  if (p.resident) {
    for (int lb = 0; lb < nb; ++lb) {
      const uint32_t n = s_ce[lb] - s_cb[lb];
      for (uint32_t i = tid; i < n; i += blockDim.x) {
        ChunkDesc cd = p.chunks[s_src_c[lb] + i];
        cd.cw_off = cd.cw_off - s_src_cw[lb] + s_dst_cw[lb];
        cd.val_off = cd.val_off - s_src_v[lb] + s_dst_v[lb];
        s_ch[s_cb[lb] + i] = cd;
      }
      for (uint32_t i = tid; i < s_n_cw[lb]; i += blockDim.x) s_cw[s_dst_cw[lb] + i] = p.colwords[s_src_cw[lb] + i];
      for (uint32_t i = tid; i < s_n_v[lb]; i += blockDim.x) s_val[s_dst_v[lb] + i] = p.vals[s_src_v[lb] + i];
    }
    v.ch = s_ch; v.cw = s_cw; v.vals = s_val;
  }
  __syncthreads();
  return v;
}

// Band x vector for work item (local band lb, k-split part ks_i): partial[(lb*ks + ks_i)*BH + row].
template <int BH>
__device__ __forceinline__ void band_gemv(const BandView& v, const float* hs, float* partial, int lb, int ks_i, int ks,
                                          int lane) {
  float acc[BH];
#pragma unroll
  for (int r = 0; r < BH; ++r) acc[r] = 0.f;
  for (uint32_t c = v.cb[lb] + ks_i; c < v.ce[lb]; c += ks) {
    const ChunkDesc cd = v.ch[c];
    const int ncols = cd.ncols_kr & 0xFFFF;
    if (lane < ncols) {
      const uint32_t w = v.cw[cd.cw_off + lane];
      const unsigned rm = w >> 16;
      const float xv = hs[w & 0xFFFFu];
      const float* val = v.vals + cd.val_off + lane;
      int cnt = 0;
#pragma unroll
      for (int r = 0; r < BH; ++r)
        if ((rm >> r) & 1u) { acc[r] = fmaf(val[cnt * ncols], xv, acc[r]); ++cnt; }
    }
  }
  warp_reduce_rows<BH>(acc, lane);
  partial[(lb * ks + ks_i) * BH + warp_row<BH>(lane)] = acc[0];
}

__device__ __forceinline__ float gru_gate(const float* partial, const float (&bq)[3], const float (&gi)[3], int g_tri,
                                          int g_r, int ks, int BH, float hprev) {
  float q[3];
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    float s = bq[g];
    for (int k = 0; k < ks; ++k) s += partial[((g_tri * 3 + g) * ks + k) * BH + g_r];
    q[g] = s;
  }
  const float rg = sigmoidf_(gi[0] + q[0]);
  const float zg = sigmoidf_(gi[1] + q[1]);
  const float ng = tanhf(gi[2] + rg * q[2]);
  return (1.f - zg) * ng + zg * hprev;
}

// ---------------------------------------------------------------------------------------------
// cooperative-grid version (h through L2, bounded global barrier)
// ---------------------------------------------------------------------------------------------
template <int BH>
__global__ void __launch_bounds__(1024, 1) gru_recurrent_kernel(const GruParams p) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nb = 3 * p.tpc;
  float* hs = reinterpret_cast<float*>(smem);
  float* partial = hs + p.H;  // [nb][ks][BH]
  __shared__ int s_abort;
  if (tid == 0) s_abort = 0;
  const BandView v = setup_bands(p, blockIdx.x, reinterpret_cast<uint8_t*>(partial + nb * p.ks * BH));

  const int nwarps = blockDim.x >> 5;
  const bool gate_thread = tid < p.tpc * p.bh;
  const int g_tri = tid / p.bh, g_r = tid % p.bh;
  const int unit = (blockIdx.x * p.tpc + g_tri) * p.bh + g_r;
  const bool gate_live = gate_thread && unit < p.H;
  float bq[3] = {0.f, 0.f, 0.f}, bi[3] = {0.f, 0.f, 0.f};
  if (gate_live)
    for (int g = 0; g < 3; ++g) {
      bq[g] = p.b_hh[g * p.H + unit];
      if (p.b_ih) bi[g] = p.b_ih[g * p.H + unit];
    }

  for (int t = 0; t < p.T; ++t) {
    float gi[3] = {0.f, 0.f, 0.f};
    if (gate_live)
      for (int g = 0; g < 3; ++g) gi[g] = __ldg(p.gi + (int64_t)t * 3 * p.H + g * p.H + unit) + bi[g];
    // h_{t-1}: written by other blocks during this launch -> read through L2
    const float* hprev = t == 0 ? p.h0 : p.out + (int64_t)(t - 1) * p.H;
    for (int i = tid; i < p.H; i += blockDim.x) hs[i] = hprev ? __ldcg(hprev + i) : 0.f;
    __syncthreads();
    for (int item = warp; item < nb * p.ks; item += nwarps) band_gemv<BH>(v, hs, partial, item / p.ks, item % p.ks, p.ks, lane);
    __syncthreads();
    if (gate_live) {
      const float hn = gru_gate(partial, bq, gi, g_tri, g_r, p.ks, BH, hs[unit]);
      p.out[(int64_t)t * p.H + unit] = hn;
      if (p.outT) p.outT[(int64_t)unit * p.ldT + t] = hn;
      if (t == p.T - 1 && p.hT) p.hT[unit] = hn;
    }
    if (t == p.T - 1) break;
    __syncthreads();
    if (tid == 0) {
      // bounded grid-wide barrier: arrive with release, poll with acquire
      if ((int)blockIdx.x != p.skip_cta) red_release_gpu_add(p.bar, 1u);
      const unsigned target = (unsigned)(t + 1) * gridDim.x;
      unsigned spins = 0;
      while (ld_acquire_gpu(p.bar) < target) {
        if (++spins > p.spin_limit) {
          atomicExch(p.status, (unsigned)GRIM_ERR_TIMEOUT);
          s_abort = 1;
          break;
        }
      }
    }
    __syncthreads();
    if (s_abort) break;
  }
}

// ---------------------------------------------------------------------------------------------
// cluster version (h through distributed shared memory, hardware cluster barrier - no spin waits)
// ---------------------------------------------------------------------------------------------
template <int BH>
__global__ void __launch_bounds__(1024, 1) gru_cluster_kernel(const GruParams p) {
  extern __shared__ __align__(16) uint8_t smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster.block_rank();
  const int CS = (int)cluster.num_blocks();
  const int nb = 3 * p.tpc;
  const int U = p.tpc * p.bh;                      // hidden units owned by this CTA
  float* hs = reinterpret_cast<float*>(smem);      // [2][H], double-buffered h
  float* hnew = hs + 2 * p.H;                      // [U]
  float* partial = hnew + ((U + 3) & ~3);          // [nb][ks][BH]
  const BandView v = setup_bands(p, rank, reinterpret_cast<uint8_t*>(partial + nb * p.ks * BH));

  const int nwarps = blockDim.x >> 5;
  const bool gate_live = tid < U;
  const int g_tri = tid / p.bh, g_r = tid % p.bh;
  const int unit = rank * U + tid;
  float bq[3] = {0.f, 0.f, 0.f}, bi[3] = {0.f, 0.f, 0.f};
  if (gate_live)
    for (int g = 0; g < 3; ++g) {
      bq[g] = p.b_hh[g * p.H + unit];
      if (p.b_ih) bi[g] = p.b_ih[g * p.H + unit];
    }
  for (int i = tid; i < p.H; i += blockDim.x) hs[i] = p.h0 ? p.h0[i] : 0.f;
  cluster.sync();  // every CTA of the cluster is resident and has initialised its buffers

  for (int t = 0; t < p.T; ++t) {
    const float* hcur = hs + (t & 1) * p.H;
    float* hnxt_local = hs + ((t + 1) & 1) * p.H;
    float gi[3] = {0.f, 0.f, 0.f};
    if (gate_live)
      for (int g = 0; g < 3; ++g) gi[g] = __ldg(p.gi + (int64_t)t * 3 * p.H + g * p.H + unit) + bi[g];
    for (int item = warp; item < nb * p.ks; item += nwarps) band_gemv<BH>(v, hcur, partial, item / p.ks, item % p.ks, p.ks, lane);
    __syncthreads();
    if (gate_live) {
      const float hn = gru_gate(partial, bq, gi, g_tri, g_r, p.ks, BH, hcur[unit]);
      hnew[tid] = hn;
      p.out[(int64_t)t * p.H + unit] = hn;
      if (p.outT) p.outT[(int64_t)unit * p.ldT + t] = hn;
      if (t == p.T - 1 && p.hT) p.hT[unit] = hn;
    }
    __syncthreads();
    // broadcast this CTA's slice of h_t into the next-step buffer of every CTA of the cluster
    if ((U & 3) == 0) {
      const int q = U >> 2;
      for (int i = tid; i < CS * q; i += blockDim.x) {
        const int dst = i / q, j = i - dst * q;
        float4* remote = cluster.map_shared_rank(reinterpret_cast<float4*>(hnxt_local + rank * U) + j, dst);
        *remote = reinterpret_cast<const float4*>(hnew)[j];
      }
    } else {
      for (int i = tid; i < CS * U; i += blockDim.x) {
        const int dst = i / U, j = i - dst * U;
        *cluster.map_shared_rank(hnxt_local + rank * U + j, dst) = hnew[j];
      }
    }
    cluster.sync();  // release our stores, acquire everyone else's; also keeps all CTAs alive until the end
  }
}

// ---------------------------------------------------------------------------------------------
// cluster version with W_hh in registers.  Every warp keeps its share of the bands in registers for the whole
// sequence, and the new state travels by asynchronous shared-memory stores counted on mbarriers instead of through a
// cluster barrier (whose release / acquire pair was the largest stall of a step): a band is cut into ks parts (work items),
// an item's kept columns are dealt to S slots x 32 lanes, and a lane holds per slot the column index and
// the column's BH values expanded to row positions (zeros where the row is not kept).  A time step then
// costs one shared-memory gather of h and BH / 2 packed FMAs (two rows each) per slot - no index decoding, no predicates.
// NI = items per warp, THREADS = the most threads a variant is launched with.  What bounds a step is a chain of latencies
// (gather, sums, reduction, gates, exchange), in which the issue of a scheduler's warps is the largest part that the shape
// decides: the variant with the fewest issued instructions per step is taken.  Shapes that need more slots than the compiled
// menu use the other kernels.  The menu's sizes are what registers hold: reloading weights every step costs more than any
// schedule gains.  (Three of the widest spill a little: <16, 1, 8, 384> 88 bytes a thread, <4, 4, 7, 384> 36, <4, 6, 8, 256> 8.)
// ---------------------------------------------------------------------------------------------
template <int BH, int NI, int S, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) gru_cluster_reg_kernel(const GruParams p) {
  extern __shared__ __align__(16) float smem_f[];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster.block_rank();
  const int CS = (int)cluster.num_blocks();
  const int nb = 3 * p.tpc;
  const int U = p.tpc * p.bh;
  const int H = p.H;
  const int ks = p.ks;
  float* hs = smem_f;                          // [2][H]
  float* partial = hs + 2 * H;                 // [2][nb][ks][BH]: steps alternate, so that a warp that is ahead overwrites nothing
  const int part_len = nb * ks * BH;

  // ---- one-time: this thread's share of W_hh (built on the host when the handle was created): coalesced loads
  unsigned long long val[NI][S][BH / 2];  // pairs of neighbouring rows
  uint32_t col[NI][(S + 1) / 2];          // columns of two slots
  {
    const float2* iv = reinterpret_cast<const float2*>(p.img_val) + (size_t)rank * NI * S * (BH / 2) * THREADS + tid;
    const uint32_t* ic = p.img_col + (size_t)rank * NI * ((S + 1) / 2) * THREADS + tid;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
#pragma unroll
      for (int s = 0; s < (S + 1) / 2; ++s) col[i][s] = __ldg(ic + (size_t)(i * ((S + 1) / 2) + s) * THREADS);
#pragma unroll
      for (int s = 0; s < S; ++s)
#pragma unroll
        for (int r = 0; r < BH / 2; ++r) {
          const float2 v = __ldg(iv + (size_t)((i * S + s) * (BH / 2) + r) * THREADS);
          val[i][s][r] = walk_pair(v.x, v.y);
        }
    }
  }

  // The gates of the CTA's U hidden units are worked out by several groups of warps at once, each of which sends the new
  // values to its share of the cluster (sixteen stores one after the other by the same warp were 300 cycles of the step).
  const int wg = (U + 31) / 32, groups = min(min((int)(blockDim.x >> 5) / wg, 4), CS), group = warp / wg;
  const int gu = (warp - group * wg) * 32 + lane;
  const int g_tri = gu / p.bh, g_r = gu % p.bh;
  const int unit = rank * U + gu;
  const bool gate_live = group < groups && gu < U && unit < H;  // (the last CTA may own fewer groups of units)
  const int dst0 = CS * group / groups, dst1 = CS * (group + 1) / groups;
  const bool stores = group == groups - 1;
  float bq[3] = {0.f, 0.f, 0.f};
  float gi[3] = {0.f, 0.f, 0.f};
  float h_own = 0.f;  // the unit's state
  if (gate_live) {
    for (int g = 0; g < 3; ++g) {
      bq[g] = p.b_hh[g * H + unit];
      gi[g] = __ldg(p.gi + g * H + unit);
    }
    h_own = p.h0 ? p.h0[unit] : 0.f;
  }
  for (int i = tid; i < H; i += (int)blockDim.x) hs[i] = p.h0 ? p.h0[i] : 0.f;
  // The state exchange: the threads that own a hidden unit send its new value into the next-step buffer of every
  // CTA of the cluster with asynchronous stores that count their bytes on the receiver's mbarrier; a warp starts a
  // step when the H values of that step have been counted.  No cluster-wide barrier and no fence per step: values of a
  // step leave a CTA only after all its warps have read the state before it (the block barrier below), and a buffer is
  // written again only by CTAs that have received such values from everybody - so every CTA has to own units and send: one
  // that does not could fall two steps behind and find the bytes of two states in one phase of its barrier.
  uint64_t* hbar = reinterpret_cast<uint64_t*>(partial + 2 * part_len);  // [2], 8-byte aligned (all counts are even)
  volatile int* s_failed = reinterpret_cast<volatile int*>(hbar + 2);
  if (tid == 0) *s_failed = 0;
  if (tid == 0) {
    gru_mbar_init(hbar, 1);
    gru_mbar_init(hbar + 1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster.sync();
  const uint32_t hs_local = (uint32_t)__cvta_generic_to_shared(hs), bar_local = (uint32_t)__cvta_generic_to_shared(hbar);

  bool lost = false;  // one of this warp's waits has run out (or another warp's, before it)
  for (int t = 0; t < p.T; ++t) {
    const int cur = t & 1, nxt = cur ^ 1;
    const float* hcur = hs + cur * H;
    float* part_t = partial + cur * part_len;
    // this step's outputs arrive on the next buffer's barrier: announce the byte count (fast CTAs may already be
    // sending, which drives the count negative; the pending arrival keeps the phase open until it is announced)
    if (tid == 0 && t + 1 < p.T && !lost) gru_mbar_arrive_expect_tx(hbar + nxt, (unsigned)H * 4u);
    // pre-activations of the next step are fetched now so that their DRAM latency hides behind this step
    float gi_next[3] = {0.f, 0.f, 0.f};
    if (gate_live && t + 1 < p.T)
      for (int g = 0; g < 3; ++g) gi_next[g] = __ldg(p.gi + (int64_t)(t + 1) * 3 * H + g * H + unit);
    // RI items are multiplied and then reduced together (their exchanges overlap)
    constexpr int RI = NI * BH == 16 || NI * BH == 32 ? NI : 1;
#pragma unroll
    for (int i0 = 0; i0 < NI; i0 += RI) {
      float acc[RI * BH];
#pragma unroll
      for (int i = 0; i < RI; ++i) {
        unsigned long long sum[BH / 2];
#pragma unroll
        for (int r = 0; r < BH / 2; ++r) sum[r] = 0ull;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const uint32_t cw = col[i0 + i][s / 2];
          const float xv = hcur[(s & 1) ? cw >> 16 : cw & 0xFFFFu];
          const unsigned long long x2 = walk_pair(xv, xv);
#pragma unroll
          for (int r = 0; r < BH / 2; ++r) walk_ffma2(sum[r], val[i0 + i][s][r], x2);
        }
#pragma unroll
        for (int r = 0; r < BH / 2; ++r) {
          acc[i * BH + 2 * r] = __uint_as_float((unsigned)sum[r]);
          acc[i * BH + 2 * r + 1] = __uint_as_float((unsigned)(sum[r] >> 32));
        }
      }
      warp_reduce_rows<RI * BH>(acc, lane);
      const int at = (warp * NI + i0) * BH + warp_row<RI * BH>(lane);
      if (at < part_len) part_t[at] = acc[0];
    }
    __syncthreads();
    if (gate_live) {
      float q[3];
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        const float* part = part_t + (g_tri * 3 + g) * ks * BH + g_r;
        q[g] = bq[g] + part[0];
        for (int k = 1; k < ks; ++k) q[g] += part[k * BH];
      }
      const float rg = __frcp_rn(1.f + expf(-(gi[0] + q[0]))), zg = __frcp_rn(1.f + expf(-(gi[1] + q[1])));
      const float ng = tanh_both(gi[2] + rg * q[2]);
      h_own = (1.f - zg) * ng + zg * h_own;
      if (t + 1 < p.T && !lost) {
        // one 4-byte store per destination (pooling four neighbours' values into 16-byte stores was slower: the
        // shuffles lengthen the chain more than the fewer messages save)
        const uint32_t dst_local = hs_local + (uint32_t)(nxt * H + unit) * 4u, bar_nxt = bar_local + (uint32_t)nxt * 8u;
#pragma unroll 4
        for (int dst = dst0; dst < dst1; ++dst) gru_st_async_f32(dst_local, bar_nxt, (uint32_t)dst, h_own);
      }
      if (stores) {  // after the exchange has left: nobody waits for these
        p.out[(int64_t)t * H + unit] = h_own;
        if (p.outT) p.outT[(int64_t)unit * p.ldT + t] = h_own;
        if (t == p.T - 1 && p.hT) p.hT[unit] = h_own;
      }
    }
#pragma unroll
    for (int g = 0; g < 3; ++g) gi[g] = gi_next[g];
    if (t + 1 < p.T) {
      // the next step's state: bounded wait on the local barrier (its (t / 2)-th use), one thread of every warp.  When it
      // runs out the block goes through its remaining steps without waiting: the results are invalid and reported.  A warp that
      // knows neither announces nor sends any more (a phase that is still open takes no second announcement, and bytes that
      // nobody waits for would pile up on the others' barriers), so the others' waits run out too.  (The vote costs nothing:
      // 396 -> 385 us for two layers of 1024, 200 steps.)
      const unsigned parity = (unsigned)((t >> 1) & 1);
      if (lane == 0) {
        bool ok = false;
        if (!*s_failed)
          for (unsigned it = 0; it < p.spin_limit && !ok; ++it) {
            ok = gru_mbar_try_wait(hbar + nxt, parity);
            if (!ok && (it & 63u) == 63u && *s_failed) break;
          }
        if (__builtin_expect(!ok, 0)) {
          lost = true;
          if (!*s_failed) {
            *s_failed = 1;
            atomicExch(p.status, (unsigned)GRIM_ERR_TIMEOUT);
          }
        }
      }
      lost = __any_sync(0xffffffffu, lost);
    }
  }
  cluster.sync();  // no CTA leaves while another may still address its shared memory
}

// The same for a stack of layers in one launch: a cluster per matrix, W_hh of every layer and W_ih of the upper ones.
// Four more warps, which hold no weights (registers are dealt out again at the start), move what has to be moved through memory:
// three bring the next steps' pre-activations (or, in a cluster that projects, inputs) into shared memory, loads a step ahead
// of their use, one writes results.  They meet the others at the block barrier of every step and are otherwise off the chain.
// Clusters of a stack wait for each other value by value: buffers between them start out as kNotYet, and who finds that in
// place of a value asks again.  (Flags beside the values cost a fence per step: 2.3 us a step instead of 1.35.)  So a layer is a
// few steps behind the one below it, where launches per layer and chunk of time were a chunk and a launch behind: two layers of
// 1024, 200 steps 385 -> 298 us; three of 1024, 133 steps 332 -> 213; 20 steps of two layers 81 -> 50.
// A cluster only ever waits for one with a lower number, which needs nothing from it: whatever order they start in, all end.
constexpr int kHelperThreads = 128, kHelperRegs = 40, kAheadSlots = 4, kBringers = 96, kInFlight = 3;
template <int THREADS>
struct MainRegs {  // what the weight-holding warps of a block may have: its registers at launch without the helpers' share
  static constexpr int wgs = THREADS / 128, at_launch = 65536 / (THREADS + kHelperThreads) / 8 * 8;
  static constexpr int all = (at_launch * (wgs + 1) - kHelperRegs) / wgs / 8 * 8, value = all < 248 ? all : 248;
};
template <int BH, int NI, int S, int THREADS>
__global__ void __launch_bounds__(THREADS + kHelperThreads, 1) gru_stack_kernel(const __grid_constant__ GruStack p) {
  extern __shared__ __align__(16) float smem_f[];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int rank = (int)cluster.block_rank();
  const int CS = (int)cluster.num_blocks();
  const GruRole& role = p.role[blockIdx.x / CS];
  const bool projects = (blockIdx.x / CS) & 1;
  const int nb = 3 * p.tpc;
  const int U = p.tpc * p.bh;
  const int H = p.H;
  const int ks = p.ks;
  const int nmain = (int)blockDim.x - kHelperThreads;  // a multiple of 128
  float* hs = smem_f;                          // [2][H]: the state; of a projection: the inputs of two steps
  float* partial = hs + 2 * H;                 // [2][nb][ks][BH]: steps alternate, so that a warp that is ahead overwrites nothing
  const int part_len = nb * ks * BH;
  float* ahead = partial + 2 * part_len;       // [kAheadSlots][3][U]: pre-activations of the steps to come
  float* s_bias = ahead + kAheadSlots * 3 * U; // [3][U]: b_hh
  float* done = s_bias + 3 * U;                // [2][U]: new states, on their way to memory
  // The state exchange: the threads that own a hidden unit send its new value into the next-step buffer of every
  // CTA of the cluster with asynchronous stores that count their bytes on the receiver's mbarrier; a warp starts a
  // step when the H values of that step have been counted.  No cluster-wide barrier and no fence per step: values of a
  // step leave a CTA only after all its warps have read the state before it (the block barrier below), and a buffer is
  // written again only by CTAs that have received such values from everybody - so every CTA has to own units and send: one
  // that does not could fall two steps behind and find the bytes of two states in one phase of its barrier.
  uint64_t* hbar = reinterpret_cast<uint64_t*>(done + 2 * U + (U & 1));  // [2], 8-byte aligned (all counts are even)
  volatile int* s_failed = reinterpret_cast<volatile int*>(hbar + 2);
  if (tid == 0) {
    *s_failed = 0;
    gru_mbar_init(hbar, 1);
    gru_mbar_init(hbar + 1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  auto meet = [] { __syncthreads(); };  // all warps, once per step

  if (tid >= nmain) {
    // ------------------------------------------------------------------ helpers
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kHelperRegs));
    const int ht = tid - nmain;
    if (ht < kBringers) {
      // The first kInFlight items per lane are asked for a step before they are put down, the others (large layers) at once.  Few
      // instructions per step: the schedulers' slots are the multiply's (written with indexes recomputed this took 0.1 us of a step).
      bool lost = false;
      auto gave_up = [&](unsigned it) {
        if (it != p.spin_limit && !((it & 63u) == 63u && *s_failed)) return false;
        lost = true;
        if (!*s_failed) {
          *s_failed = 1;
          atomicExch(p.status, (unsigned)GRIM_ERR_TIMEOUT);
        }
        return true;
      };
      const bool waits = role.waits != 0;
      auto absent = [&](float v) { return waits && !lost && __float_as_uint(v) == kNotYet; };
      if (projects) {  // items: four neighbouring inputs
        auto settle = [&](float4 v, const float* src) {
          for (unsigned it = 0; absent(v.x) || absent(v.y) || absent(v.z) || absent(v.w); ++it) {
            if (gave_up(it)) break;
            v = ld_shared_values(src);
          }
          return v;
        };
        const int items = H / 4;
        float4 w[kInFlight];
        const float* src = role.in + 4 * ht;  // of the step that is asked for next
        const bool live[kInFlight] = {ht < items, ht + kBringers < items, ht + 2 * kBringers < items};
        auto ask = [&]() {
#pragma unroll
          for (int k = 0; k < kInFlight; ++k)
            if (live[k]) w[k] = ld_shared_values(src + 4 * k * kBringers);
          src += H;
        };
        auto put = [&](int t) {  // (src is a step ahead)
          float4* dst = reinterpret_cast<float4*>(hs + (t & 1) * H) + ht;
#pragma unroll
          for (int k = 0; k < kInFlight; ++k)
            if (live[k]) dst[k * kBringers] = settle(w[k], src - H + 4 * k * kBringers);
#pragma unroll 1
          for (int i = kInFlight * kBringers; i + ht < items; i += kBringers) dst[i] = settle(ld_shared_values(src - H + 4 * i), src - H + 4 * i);
        };
        ask();
        put(0);
        if (p.T > 1) ask();
        __syncwarp();
        cluster.sync();
        for (int t = 1; t <= p.T; ++t) {
          // the buffer of step t was last read before the barrier of step t - 2
          if (t < p.T) put(t);
          if (t + 1 < p.T) ask();
          __syncwarp();
          meet();
        }
      } else {  // items: the CTA's 3 x U pre-activations
        auto settle = [&](float v, const float* src) {
          for (unsigned it = 0; absent(v); ++it) {
            if (gave_up(it)) break;
            v = ld_shared_value(src);
          }
          return v;
        };
        auto from = [&](int i) {  // place in a row of `in`, or -1
          const int g = i / U, unit = rank * U + i - g * U;
          return i < 3 * U && unit < H ? g * H + unit : -1;
        };
        float w[kInFlight];
        int at[kInFlight];
#pragma unroll
        for (int k = 0; k < kInFlight; ++k) at[k] = from(ht + k * kBringers);
        const float* src = role.in;  // the row that is asked for next
        const int64_t row = 3 * (int64_t)H;
        float* dst = ahead + ht;
        int slot = 0;
        auto ask = [&]() {
#pragma unroll
          for (int k = 0; k < kInFlight; ++k)
            if (at[k] >= 0) w[k] = ld_shared_value(src + at[k]);
          src += row;
        };
        auto put = [&]() {  // (src is a row ahead)
#pragma unroll
          for (int k = 0; k < kInFlight; ++k)
            if (at[k] >= 0) dst[k * kBringers] = settle(w[k], src - row + at[k]);
#pragma unroll 1
          for (int i = kInFlight * kBringers; i + ht < 3 * U; i += kBringers)
            if (from(i + ht) >= 0) dst[i] = settle(ld_shared_value(src - row + from(i + ht)), src - row + from(i + ht));
          slot = slot + 1 == kAheadSlots ? 0 : slot + 1;
          dst = ahead + ht + slot * 3 * U;
        };
        ask();
        put();
        if (p.T > 1) ask();
        __syncwarp();
        cluster.sync();
        for (int t = 1; t <= p.T; ++t) {
          if (t < p.T) put();
          if (t + 1 < p.T) ask();
          __syncwarp();
          meet();
        }
      }
      meet();
    } else {
      // this lane's units: lane, lane + 32, ... of the CTA's (the last CTA may own fewer)
      const int units = min(U, H - rank * U);
      float* out = role.out + rank * U + lane;
      auto write_state = [&](int t) {
        const float* from = done + (t & 1) * U + lane;
#pragma unroll 1
        for (int i = 0; i + lane < units; i += 32) {
          const float v = from[i];
          st_shared_value(out + i, v);
          if (t == p.T - 1 && role.hT) role.hT[rank * U + lane + i] = v;
        }
        out += H;
      };
      cluster.sync();
      for (int t = 0; t < p.T; ++t) {
        meet();
        if (projects) {
          const float* part_t = partial + (t & 1) * part_len;
          for (int i = 0; i + lane < units; i += 32) {
            const float* part = part_t + (i + lane) / p.bh * 3 * ks * BH + (i + lane) % p.bh;
            float v[3];
#pragma unroll
            for (int g = 0; g < 3; ++g) {
              v[g] = __ldg(role.bias + g * H + rank * U + lane + i) + part[g * ks * BH];
              for (int k = 1; k < ks; ++k) v[g] += part[(g * ks + k) * BH];
            }
#pragma unroll
            for (int g = 0; g < 3; ++g) st_shared_value(out + g * H + i, v[g]);
          }
          out += 3 * H;
        } else if (t > 0) {
          write_state(t - 1);
        }
        __syncwarp();
      }
      meet();
      if (!projects) write_state(p.T - 1);
    }
    __syncwarp();
    cluster.sync();
    return;
  }

  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(MainRegs<THREADS>::value));
  // ---- one-time: this thread's share of the matrix (built on the host when the handle was created): coalesced loads
  unsigned long long val[NI][S][BH / 2];  // pairs of neighbouring rows
  uint32_t col[NI][(S + 1) / 2];          // columns of two slots
  {
    const float2* iv = reinterpret_cast<const float2*>(role.img_val) + (size_t)rank * NI * S * (BH / 2) * THREADS + tid;
    const uint32_t* ic = role.img_col + (size_t)rank * NI * ((S + 1) / 2) * THREADS + tid;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
#pragma unroll
      for (int s = 0; s < (S + 1) / 2; ++s) col[i][s] = __ldg(ic + (size_t)(i * ((S + 1) / 2) + s) * THREADS);
#pragma unroll
      for (int s = 0; s < S; ++s)
#pragma unroll
        for (int r = 0; r < BH / 2; ++r) {
          const float2 v = __ldg(iv + (size_t)((i * S + s) * (BH / 2) + r) * THREADS);
          val[i][s][r] = walk_pair(v.x, v.y);
        }
    }
  }

  // The gates of the CTA's U hidden units are worked out by several groups of warps at once, each of which sends the new
  // values to its share of the cluster (sixteen stores one after the other by the same warp were 300 cycles of the step).
  const int wg = (U + 31) / 32, groups = min(min((nmain >> 5) / wg, 4), CS), group = warp / wg;
  const int gu = (warp - group * wg) * 32 + lane;
  const int g_tri = gu / p.bh, g_r = gu % p.bh;
  const int unit = rank * U + gu;
  const bool gate_live = !projects && group < groups && gu < U && unit < H;  // (the last CTA may own fewer groups of units)
  const int dst0 = CS * group / groups, dst1 = CS * (group + 1) / groups;
  const bool keeps = group == groups - 1;  // leaves the new values for the helper that writes them to memory
  float h_own = 0.f;  // the unit's state
  if (gate_live) {
    for (int g = 0; g < 3; ++g) s_bias[g * U + gu] = role.bias[g * H + unit];
    h_own = role.h0 ? role.h0[unit] : 0.f;
  }
  if (!projects)
    for (int i = tid; i < H; i += nmain) hs[i] = role.h0 ? role.h0[i] : 0.f;
  cluster.sync();
  const uint32_t hs_local = (uint32_t)__cvta_generic_to_shared(hs), bar_local = (uint32_t)__cvta_generic_to_shared(hbar);

  bool lost = false;  // one of this warp's waits has run out (or another warp's, before it)
  for (int t = 0; t < p.T; ++t) {
    const int cur = t & 1, nxt = cur ^ 1;
    const float* hcur = hs + cur * H;
    float* part_t = partial + cur * part_len;
    // this step's outputs arrive on the next buffer's barrier: announce the byte count (fast CTAs may already be
    // sending, which drives the count negative; the pending arrival keeps the phase open until it is announced)
    if (tid == 0 && !projects && t + 1 < p.T && !lost) gru_mbar_arrive_expect_tx(hbar + nxt, (unsigned)H * 4u);
    float gi[3] = {0.f, 0.f, 0.f};  // read now, so that nothing waits for them later
    if (gate_live) {
      const float* at = ahead + (t & (kAheadSlots - 1)) * 3 * U + gu;
      gi[0] = at[0] + s_bias[gu]; gi[1] = at[U] + s_bias[U + gu]; gi[2] = at[2 * U];
    }
    // RI items are multiplied and then reduced together (their exchanges overlap)
    constexpr int RI = NI * BH == 16 || NI * BH == 32 ? NI : 1;
#pragma unroll
    for (int i0 = 0; i0 < NI; i0 += RI) {
      float acc[RI * BH];
#pragma unroll
      for (int i = 0; i < RI; ++i) {
        unsigned long long sum[BH / 2];
#pragma unroll
        for (int r = 0; r < BH / 2; ++r) sum[r] = 0ull;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const uint32_t cw = col[i0 + i][s / 2];
          const float xv = hcur[(s & 1) ? cw >> 16 : cw & 0xFFFFu];
          const unsigned long long x2 = walk_pair(xv, xv);
#pragma unroll
          for (int r = 0; r < BH / 2; ++r) walk_ffma2(sum[r], val[i0 + i][s][r], x2);
        }
#pragma unroll
        for (int r = 0; r < BH / 2; ++r) {
          acc[i * BH + 2 * r] = __uint_as_float((unsigned)sum[r]);
          acc[i * BH + 2 * r + 1] = __uint_as_float((unsigned)(sum[r] >> 32));
        }
      }
      warp_reduce_rows<RI * BH>(acc, lane);
      const int at = (warp * NI + i0) * BH + warp_row<RI * BH>(lane);
      if (at < part_len) part_t[at] = acc[0];
    }
    meet();
    if (projects) continue;
    if (gate_live) {
      float q[3];
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        const float* part = part_t + (g_tri * 3 + g) * ks * BH + g_r;
        q[g] = g == 2 ? s_bias[2 * U + gu] + part[0] : part[0];
        for (int k = 1; k < ks; ++k) q[g] += part[k * BH];
      }
      const float rg = __frcp_rn(1.f + expf(-(gi[0] + q[0]))), zg = __frcp_rn(1.f + expf(-(gi[1] + q[1])));
      const float ng = tanh_both(gi[2] + rg * q[2]);
      h_own = (1.f - zg) * ng + zg * h_own;
      if (t + 1 < p.T && !lost) {
        // one 4-byte store per destination (pooling four neighbours' values into 16-byte stores was slower: the
        // shuffles lengthen the chain more than the fewer messages save)
        const uint32_t dst_local = hs_local + (uint32_t)(nxt * H + unit) * 4u, bar_nxt = bar_local + (uint32_t)nxt * 8u;
#pragma unroll 4
        for (int dst = dst0; dst < dst1; ++dst) gru_st_async_f32(dst_local, bar_nxt, (uint32_t)dst, h_own);
      }
      if (keeps) done[cur * U + gu] = h_own;
    }
    if (t + 1 < p.T) {
      // the next step's state: bounded wait on the local barrier (its (t / 2)-th use), one thread of every warp.  When it
      // runs out the block goes through its remaining steps without waiting: the results are invalid and reported.  A warp that
      // knows neither announces nor sends any more (a phase that is still open takes no second announcement, and bytes that
      // nobody waits for would pile up on the others' barriers), so the others' waits run out too.  (The vote costs nothing:
      // 396 -> 385 us for two layers of 1024, 200 steps.)
      const unsigned parity = (unsigned)((t >> 1) & 1);
      if (lane == 0) {
        bool ok = false;
        if (!*s_failed)
          for (unsigned it = 0; it < p.spin_limit && !ok; ++it) {
            ok = gru_mbar_try_wait(hbar + nxt, parity);
            if (!ok && (it & 63u) == 63u && *s_failed) break;
          }
        if (__builtin_expect(!ok, 0)) {
          lost = true;
          if (!*s_failed) {
            *s_failed = 1;
            atomicExch(p.status, (unsigned)GRIM_ERR_TIMEOUT);
          }
        }
      }
      lost = __any_sync(0xffffffffu, lost);
    }
  }
  meet();
  if (*s_failed) ptx::let_copies_land();
  cluster.sync();  // no CTA leaves while another may still address its shared memory
}

size_t smem_bytes(const grim_gru* g, const ModeCfg& m, int BH, bool cluster) {
  const int nb = 3 * m.tpc;
  size_t b = (size_t)nb * m.ks * BH * 4;
  if (cluster) b += (size_t)2 * g->H * 4 + (size_t)((m.tpc * g->bh + 3) & ~3) * 4;
  else b += (size_t)g->H * 4;
  if (m.resident) b += (size_t)m.max_chunks * sizeof(ChunkDesc) + (size_t)m.max_cw * 4 + (size_t)m.max_vals * 4;
  return (b + 15) & ~size_t(15);
}

template <int BH>
cudaError_t launch_grid(const grim_gru* g, const GruParams& p, cudaStream_t s) {
  const ModeCfg& m = g->grid;
  auto kern = gru_recurrent_kernel<BH>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m.smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0, sms = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, m.threads, m.smem);
  if (e != cudaSuccess) return e;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device);
  if ((int64_t)per_sm * sms < m.ctas) return cudaErrorCooperativeLaunchTooLarge;
  void* args[] = {(void*)&p};
  e = cudaLaunchCooperativeKernel((void*)kern, dim3(m.ctas), dim3(m.threads), args, m.smem, s);
  count_launch();
  return e;
}

// Once, when the handle is created (the kernel keeps them).
template <typename Kern>
cudaError_t cluster_attributes(Kern kern, const ModeCfg& m) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m.smem);
  if (e == cudaSuccess && m.ctas > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <typename Kern>
cudaError_t cluster_launch_config(Kern kern, const ModeCfg& m, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr,
                                  cudaStream_t s, bool set_attributes, int clusters = 1) {
  if (set_attributes) {
    const cudaError_t e = cluster_attributes(kern, m);
    if (e != cudaSuccess) return e;
  }
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(m.ctas * clusters);
  cfg->blockDim = dim3(m.threads);
  cfg->dynamicSmemBytes = m.smem;
  cfg->stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = m.ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  return cudaSuccess;
}

// How many clusters of this shape can be resident?  (asked once, at creation)
template <typename Kern>
int clusters_that_fit(Kern kern, const ModeCfg& m) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  if (cluster_launch_config(kern, m, &cfg, attr, nullptr, true) != cudaSuccess) { cudaGetLastError(); return 0; }
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}

template <typename Kern, typename Params>
cudaError_t launch_cluster(Kern kern, const ModeCfg& m, const Params& p, cudaStream_t s, int clusters = 1) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = cluster_launch_config(kern, m, &cfg, attr, s, false, clusters);
  if (e != cudaSuccess) return e;
  e = cudaLaunchKernelEx(&cfg, kern, p);
  count_launch();
  return e;
}

// The compiled variants of the register-resident kernel.
using GruKernel = void (*)(const GruParams);
using StackKernel = void (*)(const GruStack);
struct RegVariant {
  int BH, ni, s, threads;
  GruKernel kern;
  StackKernel stack;
};
#define GRIM_GRU_VARIANT(BH, NI, S, TH) {BH, NI, S, TH, gru_cluster_reg_kernel<BH, NI, S, TH>, gru_stack_kernel<BH, NI, S, TH>}
const RegVariant kRegVariants[] = {
    GRIM_GRU_VARIANT(8, 1, 2, 512),
    GRIM_GRU_VARIANT(8, 1, 4, 768),
    GRIM_GRU_VARIANT(8, 2, 6, 384),
    GRIM_GRU_VARIANT(8, 3, 8, 256),
    GRIM_GRU_VARIANT(4, 1, 2, 768),
    GRIM_GRU_VARIANT(4, 1, 4, 768),
    GRIM_GRU_VARIANT(4, 2, 4, 384),
    GRIM_GRU_VARIANT(4, 4, 4, 384),
    GRIM_GRU_VARIANT(4, 4, 6, 384),
    GRIM_GRU_VARIANT(4, 4, 7, 384),
    GRIM_GRU_VARIANT(4, 6, 8, 256),
    GRIM_GRU_VARIANT(16, 1, 2, 512),
    GRIM_GRU_VARIANT(16, 1, 4, 512),
    GRIM_GRU_VARIANT(16, 1, 6, 384),
    GRIM_GRU_VARIANT(16, 1, 8, 384)};
GruKernel smem_cluster_kernel(int BH) {
  return BH == 4 ? gru_cluster_kernel<4> : (BH == 8 ? gru_cluster_kernel<8> : gru_cluster_kernel<16>);
}

// Largest number of kept columns in a band, over all bands of the matrices.
int max_band_columns(const std::vector<const grim_bcr*>& mats) {
  int mx = 0;
  for (const grim_bcr* w : mats)
    for (int64_t band = 0; band < w->nbr; ++band) {
      int n = 0;
      for (int64_t j = 0; j < w->nbc; ++j) {
        const HostBlock& hb = w->blocks[(size_t)(band * w->nbc + j)];
        n += hb.kr ? hb.kc : 0;
      }
      mx = std::max(mx, n);
    }
  return mx;
}

// How much of the chunk layout the busiest CTA would hold when CTA c owns groups [c*tpc, (c+1)*tpc).
void residency_needs(const grim_gru* g, ModeCfg& m) {
  const int ntri = (int)(g->H / g->bh);
  const int nb = 3 * m.tpc;
  for (size_t l = 0; l < g->Whh.size(); ++l) {
    const grim_bcr* wh = g->Whh[l];
    std::vector<uint32_t> pos_of_band((size_t)wh->nbr);
    for (size_t p = 0; p < pos_of_band.size(); ++p) pos_of_band[wh->band_order[p]] = (uint32_t)p;
    for (int c = 0; c < m.ctas; ++c) {
      uint32_t nc = 0, ncw = 0, nv = 0;
      for (int lb = 0; lb < nb; ++lb) {
        const int tri = c * m.tpc + lb / 3;
        if (tri >= ntri) continue;
        const uint32_t pos = pos_of_band[(size_t)((lb % 3) * ntri + tri)];
        for (uint32_t k = wh->h_gemv_band_ptr[pos]; k < wh->h_gemv_band_ptr[pos + 1]; ++k) {
          const uint32_t nk = wh->h_chunks[k].ncols_kr;
          ++nc; ncw += 32; nv += (nk & 0xFFFFu) * (nk >> 16);
        }
      }
      m.max_chunks = std::max(m.max_chunks, nc);
      m.max_cw = std::max(m.max_cw, ncw);
      m.max_vals = std::max(m.max_vals, nv);
    }
  }
}

void destroy(grim_gru* g) {
  if (!g) return;
  for (float* p : g->d_bih) cudaFree(p);
  for (float* p : g->d_bhh) cudaFree(p);
  for (uint32_t* p : g->d_pos_of_band) cudaFree(p);
  for (uint32_t* p : g->d_pos_of_band_ih) cudaFree(p);
  for (float* p : g->d_img_val) cudaFree(p);
  for (uint32_t* p : g->d_img_col) cudaFree(p);
  cudaFree(g->d_never);
  for (cudaEvent_t e : g->ev) cudaEventDestroy(e);
  for (float* p : g->d_gi) cudaFree(p);
  for (cudaStream_t st : g->lstream) cudaStreamDestroy(st);
  for (cudaStream_t st : g->pstream) cudaStreamDestroy(st);
  for (cudaEvent_t e : g->ev_chunk) cudaEventDestroy(e);
  for (cudaEvent_t e : g->ev_proj) cudaEventDestroy(e);
  if (g->ev_fork) cudaEventDestroy(g->ev_fork);
  cudaFree(g->d_seq[0]);
  cudaFree(g->d_seq[1]);
  cudaFree(g->d_seqT[0]);
  cudaFree(g->d_seqT[1]);
  cudaFree(g->d_xT);
  cudaFree(g->d_sync);
  delete g;
}

constexpr size_t kSmemLimit = 200 * 1024;

}  // namespace

namespace {
// out[k * ld + t] = in[t * K + k]: the caller's T x K input, feature-major.  Blocks past the input's (blockIdx.y >= kblocks) fill the
// buffers between the clusters of a stacked launch with kNotYet.
struct FillArgs {
  uint4* at[2 * kMaxStack - 2];
  int64_t n[2 * kMaxStack - 2];  // 16-byte pieces
};
__global__ void transpose_input_kernel(const float* __restrict__ in, float* __restrict__ out, int64_t T, int64_t K, int64_t ld, int kblocks,
                                       const __grid_constant__ FillArgs fill) {
  if ((int)blockIdx.y >= kblocks) {
    const int64_t blocks = (int64_t)gridDim.x * (gridDim.y - kblocks), block = (int64_t)(blockIdx.y - kblocks) * gridDim.x + blockIdx.x;
#pragma unroll
    for (int b = 0; b < 2 * kMaxStack - 2; ++b)
      for (int64_t i = block * 256 + threadIdx.y * 32 + threadIdx.x; i < fill.n[b]; i += blocks * 256) fill.at[b][i] = make_uint4(kNotYet, kNotYet, kNotYet, kNotYet);
    return;
  }
  __shared__ float tile[32][33];
  const int64_t t0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int64_t t = t0 + i, k = k0 + threadIdx.x;
    tile[i][threadIdx.x] = (t < T && k < K) ? in[t * K + k] : 0.f;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int64_t k = k0 + i, t = t0 + threadIdx.x;
    if (k < K && t < T) out[k * ld + t] = tile[threadIdx.x][i];
  }
}
// Records the next timing event of the pool on stream s (profiling only).
void profile_mark(grim_gru* g, int kind, cudaStream_t s) {
  if (g->ev_used >= (int)g->ev.size()) return;
  g->ev_kind[(size_t)g->ev_used] = kind;
  cudaEventRecord(g->ev[(size_t)g->ev_used++], s);
}
}  // namespace

extern "C" grim_status_t grim_gru_create(int layers, const grim_bcr_t* W_ih, const grim_bcr_t* W_hh,
                                         const float* const* b_ih, const float* const* b_hh, int64_t max_T,
                                         grim_gru_t* out) {
  if (layers <= 0 || !W_ih || !W_hh || !b_ih || !b_hh || !out || max_T <= 0) return GRIM_ERR_INVALID_ARG;
  for (int l = 0; l < layers; ++l)
    if (!W_ih[l] || !W_hh[l] || !b_ih[l] || !b_hh[l]) return GRIM_ERR_INVALID_ARG;
  const int64_t H = W_hh[0]->K;
  const int bh = W_hh[0]->bh;
  for (int l = 0; l < layers; ++l) {
    const grim_bcr *wi = W_ih[l], *wh = W_hh[l];
    if (wi->device < 0 || wh->device < 0) return GRIM_ERR_INVALID_ARG;
    if (wh->K != H || wh->M != 3 * H || wi->M != 3 * H) return GRIM_ERR_SHAPE;
    if (l > 0 && wi->K != H) return GRIM_ERR_SHAPE;
    if (wi->dtype != GRIM_F32 || wh->dtype != GRIM_F32) return GRIM_ERR_DTYPE;
    if (wh->bh != bh || H % bh != 0 || !wh->gemv_ok) return GRIM_ERR_UNSUPPORTED;
    if (H % 4 != 0) return GRIM_ERR_UNSUPPORTED;  // rows of 3H floats are filled and read as 16-byte vectors
  }
  grim_gru* g = new (std::nothrow) grim_gru();
  if (!g) return GRIM_ERR_ALLOC;
  g->L = layers; g->H = H; g->max_T = max_T; g->bh = bh;
  cudaGetDevice(&g->device);
  const int ntri = (int)(H / bh);
  const int BHc = bh <= 4 ? 4 : (bh <= 8 ? 8 : 16);
  grim_status_t st = GRIM_OK;
  try {
    for (int l = 0; l < layers && st == GRIM_OK; ++l) {
      const grim_bcr* wh = W_hh[l];
      g->Wih.push_back(W_ih[l]);
      g->Whh.push_back(wh);
      std::vector<uint32_t> pos_of_band((size_t)wh->nbr);
      for (size_t p = 0; p < pos_of_band.size(); ++p) pos_of_band[wh->band_order[p]] = (uint32_t)p;
      const grim_bcr* wi = W_ih[l];
      std::vector<uint32_t> pos_ih((size_t)wi->nbr);
      for (size_t p = 0; p < pos_ih.size(); ++p) pos_ih[wi->band_order[p]] = (uint32_t)p;
      float *db1 = nullptr, *db2 = nullptr;
      uint32_t *dp = nullptr, *dpi = nullptr;
      cudaError_t e = cudaMalloc((void**)&db1, (size_t)3 * H * 4);
      if (e == cudaSuccess) { g->d_bih.push_back(db1); e = cudaMalloc((void**)&db2, (size_t)3 * H * 4); }
      if (e == cudaSuccess) { g->d_bhh.push_back(db2); e = cudaMalloc((void**)&dp, pos_of_band.size() * 4); }
      if (e == cudaSuccess) { g->d_pos_of_band.push_back(dp); e = cudaMalloc((void**)&dpi, pos_ih.size() * 4); }
      if (e == cudaSuccess) {
        g->d_pos_of_band_ih.push_back(dpi);
        e = cudaMemcpy(dpi, pos_ih.data(), pos_ih.size() * 4, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(db1, b_ih[l], (size_t)3 * H * 4, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(db2, b_hh[l], (size_t)3 * H * 4, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(dp, pos_of_band.data(), pos_of_band.size() * 4, cudaMemcpyHostToDevice);
      }
      if (e != cudaSuccess) st = e == cudaErrorMemoryAllocation ? GRIM_ERR_ALLOC : GRIM_ERR_CUDA;
    }
    if (st == GRIM_OK) {
      cudaError_t e = cudaSuccess;
      for (int l = 0; l < layers && e == cudaSuccess; ++l) {
        float* p = nullptr;
        e = cudaMalloc((void**)&p, (size_t)max_T * 3 * H * 4);
        if (e == cudaSuccess) g->d_gi.push_back(p);
      }
      g->d_gi_saved.resize(g->d_gi.size());  // sized here so that grim_gru_seq_static never touches the heap
      for (int i = 0; i < 2 * (layers - 1) && e == cudaSuccess; ++i) {
        cudaStream_t st = nullptr;
        e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
        if (e == cudaSuccess) (i & 1 ? g->pstream : g->lstream).push_back(st);
      }
      for (int i = 0; i < 2 * layers * g->max_chunks && e == cudaSuccess; ++i) {
        cudaEvent_t ev = nullptr;
        e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e == cudaSuccess) (i & 1 ? g->ev_proj : g->ev_chunk).push_back(ev);
      }
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g->ev_fork, cudaEventDisableTiming);
      if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_seq[0], (size_t)max_T * H * 4);
      if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_seq[1], (size_t)max_T * H * 4);
      const size_t ldT_max = (size_t)((max_T + 3) / 4 * 4);
      if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_seqT[0], ldT_max * H * 4);
      if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_seqT[1], ldT_max * H * 4);
      if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_xT, ldT_max * (size_t)W_ih[0]->K * 4);
      if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_sync, (size_t)(layers + 1) * 4);
      if (e == cudaSuccess) e = cudaMemset(g->d_sync, 0, (size_t)(layers + 1) * 4);
      if (e != cudaSuccess) st = e == cudaErrorMemoryAllocation ? GRIM_ERR_ALLOC : GRIM_ERR_CUDA;
    }
    if (st == GRIM_OK) {
      // ---- cooperative-grid shape: up to 128 CTAs, weights on-chip if they fit, else streamed from L2
      ModeCfg& m = g->grid;
      m.tpc = (ntri + 127) / 128;
      if (3 * m.tpc <= kMaxLocalBands) {
        m.ctas = (ntri + m.tpc - 1) / m.tpc;
        const int nb = 3 * m.tpc;
        m.ks = std::max(1, std::min(4, 32 / nb));
        m.threads = std::min(1024, std::max(nb * m.ks * 32, ((m.tpc * bh + 31) / 32) * 32));
        residency_needs(g, m);
        m.resident = 1;
        m.smem = smem_bytes(g, m, BHc, false);
        if (m.smem > kSmemLimit) { m.resident = 0; m.smem = smem_bytes(g, m, BHc, false); }
        m.ok = m.smem <= kSmemLimit;
      }
      // ---- cluster shape: the largest cluster (<= 16 CTAs) that divides the unit groups evenly
      for (int cs = 16; cs >= 1 && !g->cluster.ok; cs >>= 1) {
        if (ntri % cs) continue;
        ModeCfg t;
        t.tpc = ntri / cs;
        if (3 * t.tpc > kMaxLocalBands || t.tpc * bh > 1024) continue;
        t.ctas = cs;
        const int nb = 3 * t.tpc;
        t.ks = std::max(1, std::min(4, 32 / nb));
        t.threads = std::min(1024, std::max(std::max(nb * t.ks * 32, ((t.tpc * bh + 31) / 32) * 32), 256));
        residency_needs(g, t);
        t.resident = 1;
        t.smem = smem_bytes(g, t, BHc, true);
        if (t.smem > kSmemLimit) continue;  // the cluster scheme is only used with weights on-chip
        g->cluster = t;
        g->cluster.ok = clusters_that_fit(smem_cluster_kernel(BHc), g->cluster) >= 1;
        if (!g->cluster.ok) g->cluster = ModeCfg{};
      }
      // ---- register-resident cluster shapes: for W_hh, and where all layers run in one launch for W_hh and the upper layers' W_ih
      struct Candidate { double cost; const RegVariant* v; ModeCfg shape, stack; };
      // variants that hold bands of max_cols columns on clusters of cs blocks, in the order of their costs (asking whether one fits costs
      // more than all else here)
      auto candidates = [&](int max_cols, int cs, bool stack) {
        std::vector<Candidate> cands;
        // (only CTAs that own units: the exchange's flow control rests on every CTA sending in every step)
        const int tpc = (ntri + cs - 1) / cs, live = (ntri + tpc - 1) / tpc, nb = 3 * tpc, units = tpc * bh;
        for (const RegVariant& v : kRegVariants)
          for (int ks = 1; ks <= 8; ks *= 2) {
            const int items = nb * ks, warps = (items + v.ni - 1) / v.ni;
            if (v.BH != BHc || 32 * v.s * ks < max_cols + ks - 1 || std::max(32 * warps, (units + 31) / 32 * 32) > v.threads) continue;
            // issue of a scheduler's share, then the items that a warp works off one after the other (1024 units, 8 x 32:
            // 12 warps x 2 items 327 us for 200 steps, 8 x 3 items 325, 16 x 3 half items 361)
            const double cost = (double)items * (v.s * (3 + BHc / 2) + 4 * BHc + 10) / 4 + v.ni * 20;
            const size_t words = (size_t)2 * H + (size_t)2 * nb * ks * BHc;
            ModeCfg t;
            t.ctas = live; t.ks = ks; t.tpc = tpc; t.resident = 1;
            t.threads = std::max(32 * warps, std::max((units + 31) / 32 * 32, 128));
            t.smem = ((words * 4 + 15) & ~size_t(15)) + 32;  // + the two state barriers and a flag
            ModeCfg u = t;
            u.threads = (t.threads + 127) / 128 * 128 + kHelperThreads;  // whole warpgroups
            // + pre-activations ahead and biases, states to be written
            u.smem = (((words + (size_t)(kAheadSlots + 1) * 3 * units + 2 * (size_t)units + 1) * 4 + 15) & ~size_t(15)) + 32;
            if ((stack ? u.smem : t.smem) <= kSmemLimit) cands.push_back({cost, &v, t, u});
          }
        std::stable_sort(cands.begin(), cands.end(), [](const Candidate& x, const Candidate& y) { return x.cost < y.cost; });
        return cands;
      };
      // One launch for all layers: if a variant holds all matrices, as many clusters run at once, and its steps are not much longer than
      // W_hh's own variant would make them (costs; steps against those of layers chunk by chunk, us: 752 and 632: 1.69 and 2.29; 384 and
      // 285: 1.68 and 1.75; 354 and 230: 2.14 and 2.06; 648 and 188: 2.40 and 1.58).  More than three layers: layers l and l + 2 share a buffer.
      constexpr double kLongerSteps = 1.4;
      bool stack = layers > 1 && layers <= kMaxStack;
      for (int l = 1; l < layers; ++l) stack = stack && W_ih[l]->bh == bh;
      const std::vector<const grim_bcr*> upper(g->Wih.begin() + 1, g->Wih.end());
      const int cols_hh = max_band_columns(g->Whh), cols_all = stack ? std::max(cols_hh, max_band_columns(upper)) : 0;
      Candidate hh{}, all{};
      for (int cs = 16; cs >= 1 && !hh.v && H <= 65536; cs >>= 1) {
        const std::vector<Candidate> own = candidates(cols_hh, cs, false);
        if (stack && !own.empty())
          for (const Candidate& c : candidates(cols_all, cs, true)) {
            if (c.cost > kLongerSteps * own[0].cost) break;
            if (clusters_that_fit(c.v->stack, c.stack) >= 2 * layers - 1) { all = c; break; }
          }
        for (const Candidate& c : own)
          // (where the blocks with helpers fit, those without do)
          if (c.v == all.v && c.shape.ks == all.shape.ks ? cluster_attributes(c.v->kern, c.shape) == cudaSuccess : clusters_that_fit(c.v->kern, c.shape) >= 1) {
            hh = c;
            break;
          }
        if (!hh.v) all = Candidate{};
      }
      if (hh.v) {
        g->regc = hh.shape; g->regc.ok = true; g->reg_kern = hh.v->kern;
        // register images: for every thread of every CTA the columns it owns (global index + values at row positions); threads
        // are numbered with the variant's stride
        struct Image { std::vector<float> val; std::vector<uint32_t> col; };
        struct ColRec { uint32_t col, rowmask, kc; const float* v; };  // kept row a (of rowmask) has v[a * kc]
        auto image_of = [&](const grim_bcr* wh, const Candidate& c) {  // empty: does not fit
          const int NI = c.v->ni, S = c.v->s, S2 = (S + 1) / 2, TH = c.v->threads, ks = c.shape.ks, tpc = c.shape.tpc, cs = c.shape.ctas, nbb = 3 * tpc;
          Image im{std::vector<float>((size_t)cs * NI * S * BHc * TH), std::vector<uint32_t>((size_t)cs * NI * S2 * TH)};
          std::vector<float>& iv = im.val;
          std::vector<uint32_t>& ic = im.col;
          std::vector<ColRec> cols, dealt;
          std::vector<size_t> before;  // columns dealt before each round
          for (int rank = 0; rank < cs; ++rank)
            for (int lb = 0; lb < nbb; ++lb) {
              if (rank * tpc + lb / 3 >= ntri) continue;
              const int64_t band = (int64_t)(lb % 3) * ntri + (int64_t)rank * tpc + lb / 3;
              cols.clear();
              for (int64_t j = 0; j < wh->nbc; ++j) {
                const HostBlock& hb = wh->blocks[(size_t)(band * wh->nbc + j)];
                if (!(hb.kr && hb.kc)) continue;
                int bidx = 0;
                for (int c = 0; c < wh->bw; ++c) {
                  if (!((hb.colmask >> c) & 1ull)) continue;
                  cols.push_back({(uint32_t)(j * wh->bw + c), hb.rowmask, hb.kc, &wh->vals[(size_t)hb.val_off + (size_t)bidx]});
                  ++bidx;
                }
              }
              const size_t n = cols.size();
              for (int part = 0; part < ks; ++part) {
                const int item = lb * ks + part, warp = item / NI, i = item % NI;
                const size_t c0 = n * part / ks, c1 = n * (part + 1) / ks;
                // dealt so that the 32 columns of a slot fall into different shared-memory banks as far as they go (any 32 of
                // a thousand meet three or four to a bank): one from every bank's pile in turn, the longest piles first
                size_t size[32] = {}, place[32];
                int bank[32];
                for (size_t ci = c0; ci < c1; ++ci) ++size[cols[ci].col % 32];
                std::iota(bank, bank + 32, 0);
                std::stable_sort(bank, bank + 32, [&](int x, int y) { return size[x] > size[y]; });
                // column number r of a pile comes after those of earlier rounds and, in its round, of longer piles
                dealt.resize(c1 - c0);
                size_t taken[32] = {};
                for (int b = 0; b < 32; ++b) place[bank[b]] = (size_t)b;
                const size_t rounds = size[bank[0]];
                before.assign(rounds + 1, 0);
                for (int b = 0; b < 32; ++b)
                  for (size_t r = 0; r < size[b]; ++r) ++before[r + 1];
                for (size_t r = 0; r < rounds; ++r) before[r + 1] += before[r];
                for (size_t ci = c0; ci < c1; ++ci) {
                  const int b = (int)(cols[ci].col % 32);
                  dealt[before[taken[b]++] + place[b]] = cols[ci];
                }
                for (size_t k = 0; k < dealt.size(); ++k) {
                  const ColRec& cr = dealt[k];
                  const int sl = (int)(k / 32), tid = warp * 32 + (int)(k % 32);
                  if (sl >= S || tid >= TH) return Image{};
                  ic[((size_t)(rank * NI + i) * S2 + sl / 2) * TH + tid] |= cr.col << (16 * (sl & 1));
                  const float* v = cr.v;
                  for (uint32_t rm = cr.rowmask; rm; rm &= rm - 1, v += cr.kc) {
                    const int r = __builtin_ctz(rm);
                    iv[((((size_t)(rank * NI + i) * S + sl) * (BHc / 2) + r / 2) * TH + tid) * 2 + (r & 1)] = *v;
                  }
                }
              }
            }
          return im;
        };
        // (a thread per image: most of the time that creating a model takes)
        std::vector<std::future<Image>> images;
        for (const grim_bcr* w : g->Whh) images.push_back(std::async(image_of, w, hh));
        if (all.v) {
          g->stack = all.stack; g->stack.ok = true; g->stack_kern = all.v->stack;
          g->stack_hh = 0;
          if (all.v != hh.v || all.shape.ks != hh.shape.ks) {  // (of another variant)
            g->stack_hh = (int)images.size();
            for (const grim_bcr* w : g->Whh) images.push_back(std::async(image_of, w, all));
          }
          g->stack_ih = (int)images.size() - 1;  // (none for layer 0)
          for (const grim_bcr* w : upper) images.push_back(std::async(image_of, w, all));
        }
        for (std::future<Image>& f : images) {
          const Image im = f.get();
          if (st == GRIM_OK && im.val.empty()) st = GRIM_ERR_UNSUPPORTED;
          if (st != GRIM_OK) continue;
          float* dv = nullptr;
          uint32_t* dc = nullptr;
          cudaError_t e = cudaMalloc((void**)&dv, im.val.size() * 4);
          if (e == cudaSuccess) { g->d_img_val.push_back(dv); e = cudaMalloc((void**)&dc, im.col.size() * 4); }
          if (e == cudaSuccess) { g->d_img_col.push_back(dc); e = cudaMemcpy(dv, im.val.data(), im.val.size() * 4, cudaMemcpyHostToDevice); }
          if (e == cudaSuccess) e = cudaMemcpy(dc, im.col.data(), im.col.size() * 4, cudaMemcpyHostToDevice);
          if (e != cudaSuccess) st = e == cudaErrorMemoryAllocation ? GRIM_ERR_ALLOC : GRIM_ERR_CUDA;
        }
      }
      if (st == GRIM_OK && !g->grid.ok && !g->cluster.ok && !g->regc.ok) st = GRIM_ERR_UNSUPPORTED;
    }
  } catch (const std::bad_alloc&) {
    st = GRIM_ERR_ALLOC;
  }
  if (st != GRIM_OK) { cudaGetLastError(); destroy(g); return st; }
  *out = g;
  return GRIM_OK;
}

extern "C" grim_status_t grim_gru_seq(grim_gru_t g, const float* x, int64_t T, const float* h0, float* y, float* hT,
                                      grim_stream_t stream) {
  if (!g || !x || !y || T <= 0) return GRIM_ERR_INVALID_ARG;
  if (T > g->max_T) return GRIM_ERR_SHAPE;
  cudaStream_t s0 = (cudaStream_t)stream;
  g->last_stream = s0;
  const int64_t H = g->H;
  const int L = g->L;
  // preference: weights in registers > cooperative grid > shared-memory cluster
  const bool want_grid = g->force_grid && g->grid.ok;
  const bool use_reg = g->regc.ok && !want_grid;
  const bool use_cluster = !use_reg && g->cluster.ok && !g->grid.ok;
  const ModeCfg& m = use_reg ? g->regc : (use_cluster ? g->cluster : g->grid);
  const int BHc = g->bh <= 4 ? 4 : (g->bh <= 8 ? 8 : 16);
  if (cudaMemsetAsync(g->d_sync, 0, (size_t)(L + 1) * 4, s0) != cudaSuccess) return GRIM_ERR_CUDA;

  // All layers in one launch, unless they are to run in a given number of pieces or one after the other (as the static variant does,
  // whose layers share their scratch).
  // (The transposing launch then has up to kFillRows rows of blocks more than the input has: a grid has 65535.)
  constexpr int64_t kFillRows = 512;
  const bool stacked = use_reg && g->stack.ok && g->pipeline && g->want_chunks == 0 && (g->Wih[0]->K + 31) / 32 <= 65535 - kFillRows;
  // Otherwise time is cut into chunks; layer l works on chunk k while layer l - 1 works on chunk k + 1 (each layer on its own
  // stream, ordered by events), so a stack of L layers takes about (1 + (L - 1) / chunks) single-layer times instead
  // of L.  The kernels with a global barrier (fall-back) and single-layer models run as one chunk on one stream.
  int chunks = 1;
  // With four or more layers, layers l and l + 2 share an inter-layer buffer, and layer l reads its chunk-entering
  // state from that buffer while layer l + 2 may already be writing it: such stacks run one layer after the other.
  if (!stacked && g->pipeline && L > 1 && L <= 3 && (use_reg || use_cluster))
    chunks = g->want_chunks > 0 ? (int)std::min<int64_t>(g->want_chunks, T)
                                : (int)std::max<int64_t>(1, std::min<int64_t>(5, T / 25));
  const int64_t clen = ((T + chunks - 1) / chunks + 3) / 4 * 4;  // a multiple of 4: chunk starts stay 16-byte aligned
  chunks = (int)((T + clen - 1) / clen);  // the rounding may have left the last chunks empty: their events would never be recorded
  const int64_t ldT = (T + 3) / 4 * 4;
  const bool tin = g->transposed_inputs && g->d_xT != nullptr;
  auto stream_of = [&](int l) { return (chunks > 1 && l > 0) ? g->lstream[(size_t)l - 1] : s0; };
  if (chunks > 1) {
    if (cudaEventRecord(g->ev_fork, s0) != cudaSuccess) return GRIM_ERR_CUDA;
    for (int l = 1; l < L; ++l)
      if (cudaStreamWaitEvent(g->lstream[(size_t)l - 1], g->ev_fork, 0) != cudaSuccess) return GRIM_ERR_CUDA;
  }
  if (g->profile) g->ev_used = 0;
  auto launch_projection = [&](int l, const float* seq_in, int64_t t0, int64_t n, cudaStream_t s) -> grim_status_t {
    const grim_bcr* wi = g->Wih[(size_t)l];
    // gi[t, :] = W_ih x_t + b_ih for the n steps from t0 (X given q-major as n x in, output n x 3H)
    SpmmArgs a;
    a.Y = g->d_gi[(size_t)l] + t0 * 3 * H; a.ncols = n;
    a.y_sr = 1; a.y_sq = 3 * H;
    if (tin) {  // feature-major copy: a plain row-major K x n operand (fetched by TMA)
      a.X = (l == 0 ? g->d_xT : g->d_seqT[(l - 1) & 1]) + t0;
      a.x_sk = ldT; a.x_sq = 1;
    } else {
      a.X = seq_in + t0 * wi->K;
      a.x_sk = 1; a.x_sq = wi->K;
    }
    a.x_dtype = GRIM_F32; a.y_dtype = GRIM_F32;
    a.bias = g->d_bih[(size_t)l];
    if (g->profile) profile_mark(g, 0, s);
    const grim_status_t st = launch_cuda_cores(wi, a, s);
    if (g->profile) profile_mark(g, 1, s);
    return st;
  };
  auto launch_stack = [&]() -> grim_status_t {
    GruStack k = {};
    k.status = g->d_sync + L; k.H = (int)H; k.bh = g->bh; k.T = (int)T; k.tpc = g->stack.tpc; k.ks = g->stack.ks; k.spin_limit = g->spin_limit;
    for (int l = 0; l < L; ++l) {
      float* seq_out = l == L - 1 ? y : g->d_seq[l & 1];
      if (l > 0)
        k.role[2 * l - 1] = {g->d_img_val[(size_t)(g->stack_ih + l)], g->d_img_col[(size_t)(g->stack_ih + l)], g->d_bih[(size_t)l], g->d_seq[(l - 1) & 1],
                             g->d_gi[(size_t)l], nullptr, nullptr, 1};
      k.role[2 * l] = {g->d_img_val[(size_t)(g->stack_hh + l)], g->d_img_col[(size_t)(g->stack_hh + l)], g->d_bhh[(size_t)l],
                       l > 0 && g->dbg_skip_cta == kWithhold ? g->d_never : g->d_gi[(size_t)l], seq_out, h0 ? h0 + (int64_t)l * H : nullptr, hT ? hT + (int64_t)l * H : nullptr, l > 0};
    }
    if (g->profile) profile_mark(g, 2, s0);
    const cudaError_t e = launch_cluster(g->stack_kern, g->stack, k, s0, 2 * L - 1);
    if (g->profile) profile_mark(g, 3, s0);
    if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
    return GRIM_OK;
  };
  auto launch_recurrence = [&](int l, float* seq_out, int64_t t0, int64_t n, cudaStream_t s) -> grim_status_t {
    const grim_bcr* wh = g->Whh[(size_t)l];
    GruParams p;
    p.band_ptr = wh->d_gemv_band_ptr; p.chunks = wh->d_chunks; p.colwords = wh->d_colwords;
    p.vals = static_cast<const float*>(wh->d_gemv_vals); p.pos_of_band = g->d_pos_of_band[(size_t)l];
    p.b_hh = g->d_bhh[(size_t)l]; p.b_ih = nullptr; p.gi = g->d_gi[(size_t)l] + t0 * 3 * H;
    // the state entering a later chunk is the previous chunk's last output row
    p.h0 = t0 == 0 ? (h0 ? h0 + (int64_t)l * H : nullptr) : seq_out + (t0 - 1) * H;
    p.out = seq_out + t0 * H;
    p.outT = (tin && l < L - 1) ? g->d_seqT[l & 1] + t0 : nullptr;
    p.ldT = ldT;
    p.hT = (hT && t0 + n == T) ? hT + (int64_t)l * H : nullptr;
    p.bar = g->d_sync + l; p.status = g->d_sync + L;
    p.H = (int)H; p.bh = g->bh; p.T = (int)n; p.tpc = m.tpc; p.ks = m.ks; p.resident = m.resident;
    p.max_chunks = m.max_chunks; p.max_cw = m.max_cw; p.max_vals = m.max_vals;
    p.skip_cta = g->dbg_skip_cta; p.spin_limit = g->spin_limit;
    p.img_val = use_reg ? g->d_img_val[(size_t)l] : nullptr;
    p.img_col = use_reg ? g->d_img_col[(size_t)l] : nullptr;
    if (g->profile) profile_mark(g, 2, s);
    cudaError_t e;
    if (use_reg) {
      e = launch_cluster(g->reg_kern, m, p, s);
    } else if (use_cluster) {
      e = launch_cluster(smem_cluster_kernel(BHc), m, p, s);
    } else {
      if (g->bh <= 4) e = launch_grid<4>(g, p, s);
      else if (g->bh <= 8) e = launch_grid<8>(g, p, s);
      else e = launch_grid<16>(g, p, s);
    }
    if (g->profile) profile_mark(g, 3, s);
    if (e != cudaSuccess) { cudaGetLastError(); return e == cudaErrorCooperativeLaunchTooLarge ? GRIM_ERR_UNSUPPORTED : GRIM_ERR_CUDA; }
    return GRIM_OK;
  };

  // issue order: chunk-major over layers (a wavefront), so that every stream always has work queued
  for (int k = 0; k < chunks + L - 1; ++k) {
    for (int l = 0; l < L; ++l) {
      const int c = k - l;  // the chunk layer l handles in this wave
      if (c < 0 || c >= chunks) continue;
      const int64_t t0 = (int64_t)c * clen, n = std::min<int64_t>(clen, T - t0);
      if (n <= 0) continue;
      cudaStream_t s = stream_of(l);
      const float* seq_in = l == 0 ? x : g->d_seq[(l - 1) & 1];
      float* seq_out = (l == L - 1) ? y : g->d_seq[l & 1];
      grim_status_t st = GRIM_OK;
      if (stacked && l > 0) continue;
      if (l == 0) {
        if (c == 0) {  // the first layer's input is all there: one launch (after turning it feature-major)
          if (tin) {
            const int64_t K0 = g->Wih[0]->K;
            const unsigned tb = (unsigned)((T + 31) / 32), kb = (unsigned)((K0 + 31) / 32);
            FillArgs fill = {};
            int64_t pieces = 0;
            for (int b = 1; stacked && b < L; ++b) {  // (H is a multiple of 4)
              fill.at[2 * b - 2] = reinterpret_cast<uint4*>(g->d_seq[(b - 1) & 1]); fill.n[2 * b - 2] = T * H / 4;
              fill.at[2 * b - 1] = reinterpret_cast<uint4*>(g->d_gi[(size_t)b]); fill.n[2 * b - 1] = T * 3 * H / 4;
              pieces += T * H;
            }
            const unsigned fb = (unsigned)std::min<int64_t>(((pieces + 511) / 512 + tb - 1) / tb, kFillRows);  // two pieces per thread
            transpose_input_kernel<<<dim3(tb, kb + fb), dim3(32, 8), 0, s>>>(x, g->d_xT, T, K0, ldT, (int)kb, fill);
            count_launch();
          }
          st = launch_projection(0, x, 0, T, s);
        }
      } else {
        // projected on a stream of its own, so that it need not wait for the recurrence of the chunk before (2 x 1024, 200 steps: 413 -> 397 us)
        cudaStream_t ps = chunks > 1 ? g->pstream[(size_t)l - 1] : s;
        cudaEvent_t ready = g->ev_proj[(size_t)l * g->max_chunks + c];
        if (chunks > 1 && cudaStreamWaitEvent(ps, g->ev_chunk[(size_t)(l - 1) * g->max_chunks + c], 0) != cudaSuccess) return GRIM_ERR_CUDA;
        st = launch_projection(l, seq_in, t0, n, ps);
        if (st == GRIM_OK && chunks > 1 && (cudaEventRecord(ready, ps) != cudaSuccess || cudaStreamWaitEvent(s, ready, 0) != cudaSuccess)) return GRIM_ERR_CUDA;
      }
      if (st != GRIM_OK) return st;
      st = stacked ? launch_stack() : launch_recurrence(l, seq_out, t0, n, s);
      if (st != GRIM_OK) return st;
      if (chunks > 1 && cudaEventRecord(g->ev_chunk[(size_t)l * g->max_chunks + c], s) != cudaSuccess) return GRIM_ERR_CUDA;
    }
  }
  if (chunks > 1) {
    // join: the caller's stream continues when the last layer is done (lower layers finish earlier by construction,
    // but their streams are joined too so that the handle's buffers are quiescent)
    for (int l = 1; l < L; ++l)
      if (cudaStreamWaitEvent(s0, g->ev_chunk[(size_t)l * g->max_chunks + chunks - 1], 0) != cudaSuccess) return GRIM_ERR_CUDA;
  }
  return GRIM_OK;
}

extern "C" grim_status_t grim_gru_status(grim_gru_t g) {
  if (!g) return GRIM_ERR_INVALID_ARG;
  if (cudaStreamSynchronize(g->last_stream) != cudaSuccess) return GRIM_ERR_CUDA;
  unsigned v = 0;
  if (cudaMemcpy(&v, g->d_sync + g->L, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return GRIM_ERR_CUDA;
  return (grim_status_t)v;
}

// Test hook: selects the cooperative-grid kernel (the one with spin waits) whenever skip_cta >= 0 or a
// poll limit is given, makes thread block `skip_cta` stay away from its barrier and sets the number of
// polls after which a waiting block gives up.  The waits then run out and the status word reports it;
// no thread block ever waits without a bound.  skip_cta = kWithhold leaves the choice of kernel; where the layers run in one
// launch, the upper layers' pre-activations never arrive.
extern "C" grim_status_t grim_gru_debug_barrier(grim_gru_t g, int skip_cta, unsigned spin_limit) {
  if (!g) return GRIM_ERR_INVALID_ARG;
  if (skip_cta == kWithhold) {
    if (!g->stack.ok) return GRIM_ERR_UNSUPPORTED;
    const size_t bytes = (size_t)g->max_T * 3 * g->H * 4;
    if (!g->d_never && cudaMalloc((void**)&g->d_never, bytes) != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_ALLOC; }
    if (cudaMemset(g->d_never, 0xFF, bytes) != cudaSuccess) return GRIM_ERR_CUDA;  // kNotYet
    g->dbg_skip_cta = skip_cta;
    g->spin_limit = spin_limit ? spin_limit : (1u << 22);
    g->force_grid = false;
    return GRIM_OK;
  }
  if ((skip_cta >= 0 || spin_limit) && !g->grid.ok) return GRIM_ERR_UNSUPPORTED;
  g->dbg_skip_cta = skip_cta;
  g->spin_limit = spin_limit ? spin_limit : (1u << 22);
  g->force_grid = skip_cta >= 0 || spin_limit != 0;
  return GRIM_OK;
}

extern "C" grim_status_t grim_gru_set_pipeline(grim_gru_t g, int chunks) {
  if (!g || chunks < 0 || chunks > g->max_chunks) return GRIM_ERR_INVALID_ARG;
  g->pipeline = chunks != 1;
  g->want_chunks = chunks;
  return GRIM_OK;
}

extern "C" grim_status_t grim_gru_profile(grim_gru_t g, int enable) {
  if (!g) return GRIM_ERR_INVALID_ARG;
  if (enable && g->ev.empty()) {
    g->ev.resize((size_t)4 * g->L * g->max_chunks);
    g->ev_kind.assign(g->ev.size(), 0);
    for (cudaEvent_t& e : g->ev)
      if (cudaEventCreate(&e) != cudaSuccess) return GRIM_ERR_CUDA;
  }
  g->profile = enable != 0;
  g->ev_used = 0;
  return GRIM_OK;
}

extern "C" grim_status_t grim_gru_profile_read(grim_gru_t g, float* projection_ms, float* recurrent_ms) {
  if (!g || !g->profile || g->ev.empty()) return GRIM_ERR_INVALID_ARG;
  float pj = 0.f, rc = 0.f;
  for (int i = 0; i + 1 < g->ev_used; i += 2) {
    float ms = 0.f;
    if (cudaEventSynchronize(g->ev[(size_t)i + 1]) != cudaSuccess) return GRIM_ERR_CUDA;
    if (cudaEventElapsedTime(&ms, g->ev[(size_t)i], g->ev[(size_t)i + 1]) != cudaSuccess) return GRIM_ERR_CUDA;
    if (g->ev_kind[(size_t)i] == 0) pj += ms; else rc += ms;
  }
  if (projection_ms) *projection_ms = pj;
  if (recurrent_ms) *recurrent_ms = rc;
  return GRIM_OK;
}

extern "C" grim_status_t grim_gru_destroy(grim_gru_t g) {
  if (!g) return GRIM_OK;
  int cur = -1;
  const int dev = g->device;
  cudaGetDevice(&cur);
  if (cur != dev) cudaSetDevice(dev);
  destroy(g);
  if (cur != dev && cur >= 0) cudaSetDevice(cur);
  return GRIM_OK;
}

// ---------------------------------------------------------------------------------------------
// grim_gru_seq_static: the same sequence pass for callers that must not allocate device memory.
//
// The per-call scratch of the GRU pass (the hoisted pre-activations gi, T x 3H floats, and the two
// T x H buffers that carry one layer's outputs to the next) lives in a fixed array inside the
// library image instead of in buffers obtained from the CUDA allocator.  Host code cannot use the
// array's name as a device address; the address is looked up once per device with
// cudaGetSymbolAddress while that device is current, and that pointer is what the kernels receive.
// ---------------------------------------------------------------------------------------------
namespace {
constexpr size_t kStaticScratchBytes = size_t(8) << 20;  // 8 MiB, resident on every GPU that loads the library
constexpr int kMaxDevices = 64;
}  // namespace
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];
static unsigned char* g_static_scratch_addr[kMaxDevices] = {};

extern "C" grim_status_t grim_gru_seq_static(grim_gru_t g, const float* x, int64_t T, const float* h0, float* y,
                                             float* hT, grim_stream_t stream) {
  if (!g || !x || !y || T <= 0) return GRIM_ERR_INVALID_ARG;
  if (T > g->max_T) return GRIM_ERR_SHAPE;
  // carve-up of the static array: gi | seq0 | seq1, each start rounded up to 256 bytes
  auto round256 = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t gi_bytes = round256((size_t)T * 3 * (size_t)g->H * 4);
  const size_t seq_bytes = g->L > 1 ? round256((size_t)T * (size_t)g->H * 4) : 0;
  if (gi_bytes + 2 * seq_bytes > kStaticScratchBytes) return GRIM_ERR_UNSUPPORTED;  // T * H too large for 8 MiB
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return GRIM_ERR_CUDA;
  if (dev != g->device || dev < 0 || dev >= kMaxDevices) return GRIM_ERR_INVALID_ARG;
  if (!g_static_scratch_addr[dev]) {
    // one-time set-up for this device (device `dev` is current): resolve the array's device address
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return GRIM_ERR_CUDA;
    }
    g_static_scratch_addr[dev] = static_cast<unsigned char*>(p);
  }
  unsigned char* base = g_static_scratch_addr[dev];
  // Run the ordinary pass with the handle's scratch pointers pointing into the static array for the duration of
  // the call (kernel arguments are copied at launch, so the handle can be put back at once).  All layers share one
  // pre-activation buffer here, so the layers run one after the other on the caller's stream.
  std::copy(g->d_gi.begin(), g->d_gi.end(), g->d_gi_saved.begin());  // same size since creation: no allocation
  float* const saved_seq0 = g->d_seq[0];
  float* const saved_seq1 = g->d_seq[1];
  const bool saved_pipeline = g->pipeline, saved_tin = g->transposed_inputs;
  g->transposed_inputs = false;  // the feature-major copies live in allocated buffers: not used here
  for (float*& p : g->d_gi) p = reinterpret_cast<float*>(base);
  g->d_seq[0] = reinterpret_cast<float*>(base + gi_bytes);
  g->d_seq[1] = reinterpret_cast<float*>(base + gi_bytes + seq_bytes);
  g->pipeline = false;
  const grim_status_t st = grim_gru_seq(g, x, T, h0, y, hT, stream);
  std::copy(g->d_gi_saved.begin(), g->d_gi_saved.end(), g->d_gi.begin());
  g->d_seq[0] = saved_seq0;
  g->d_seq[1] = saved_seq1;
  g->pipeline = saved_pipeline;
  g->transposed_inputs = saved_tin;
  return st;
}

// -------------------------------------------------------------------------------------------------------------
// One time step for a batch of sequences (Section 6.3 times the GRU at sequence length 1 and batch 32): one launch turns
// the input and the layers' states feature-major, then one launch per layer multiplies both matrices and applies the gates.
// A thread block owns bh hidden units and 32 sequences; its 24 warps share the six bands (r, z, n of W_ih and of W_hh) that
// produce them (grim_rowwalk.cuh), their sums meet in shared memory.  (Two multiplies on batch-major operands, whose gathers
// do not coalesce, two bias passes, two clears and a gate kernel per layer took 80 us for two layers of 1024 and a batch of 32.)
// Matrices of different block heights, or without the wide layouts, take that older way, below.
// -------------------------------------------------------------------------------------------------------------
namespace {
struct StepParams {
  RowWalk w[2];               // W_ih, W_hh
  const uint32_t* pos[2];     // schedule position of every band
  const float* bias[2];
  SpmmArgs a[2];              // feature-major operands
  float* h;                   // B x H, updated in place
  float* hT;                  // null, or H x B: the new state, feature-major (input of the next layer)
  float* y;                   // null, or B x H
  int64_t B;
  int H, bh, part[2];         // warps per band
};
constexpr int kStepWarps = 24, kStepLd = 36;
template <int BH>
constexpr size_t step_smem() { return (size_t)kStepWarps * (kWalkBufFloats + BH * kStepLd) * 4; }

template <int BH>
__global__ void __launch_bounds__(kStepWarps * 32, 1) gru_step_kernel(const StepParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(16) float ssm[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int m = warp < 3 * p.part[0] ? 0 : 1, local = m ? warp - 3 * p.part[0] : warp;
  const int gate = local / p.part[m], part = local - gate * p.part[m];
  const int tri = blockIdx.x, ntri = p.H / p.bh;
  const int64_t b0 = (int64_t)blockIdx.y * 32;
  float* sums = ssm + kStepWarps * kWalkBufFloats;  // [warp][row][sequence]
  float acc1[BH];
  unsigned long long acc2[1][1];
#pragma unroll
  for (int r = 0; r < BH; ++r) acc1[r] = 0.f;
  WalkCols<1, 1> wc;
  walk_setup<1, 1, float, 0>(p.a[m], b0, lane, wc);
  const int pos = (int)__ldg(p.pos[m] + gate * ntri + tri);
  row_walk<BH, 1, 1, float, 0, false>(p.w[m], p.a[m], pos, part, p.part[m], wc, ssm + warp * kWalkBufFloats, lane, acc1, acc2,
                               [] { asm volatile("griddepcontrol.wait;" ::: "memory"); });
#pragma unroll
  for (int r = 0; r < BH; ++r) sums[(warp * BH + r) * kStepLd + lane] = acc1[r];
  __syncthreads();
  for (int i = tid; i < p.bh * 32; i += kStepWarps * 32) {
    const int r = i % p.bh, bl = i / p.bh, unit = tri * p.bh + r;  // neighbouring threads: neighbouring units of a sequence
    const int64_t b = b0 + bl;
    if (b >= p.B) continue;
    float v[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        float t = __ldg(p.bias[k] + g * p.H + unit);
        const int w0 = k * 3 * p.part[0] + g * p.part[k];
        for (int s = 0; s < p.part[k]; ++s) t += sums[((w0 + s) * BH + r) * kStepLd + bl];
        v[k][g] = t;
      }
    const int64_t at = b * p.H + unit;
    const float rg = sigmoidf_(v[0][0] + v[1][0]), zg = sigmoidf_(v[0][1] + v[1][1]);
    const float n = tanhf(v[0][2] + rg * v[1][2]);
    const float hn = (1.f - zg) * n + zg * p.h[at];
    p.h[at] = hn;
    if (p.y) p.y[at] = hn;
    if (p.hT) p.hT[(int64_t)unit * p.B + b] = hn;
  }
}

// Turns matrices of B rows feature-major: z = 0 the input (K0 columns), z > 0 the state of layer z - 1 (H columns).
constexpr int kStepMaxLayers = 16;
struct TransposeArgs {
  const float* in[kStepMaxLayers + 1];
  float* out[kStepMaxLayers + 1];
  int cols[kStepMaxLayers + 1];
};
__global__ void __launch_bounds__(256) transpose_states_kernel(const __grid_constant__ TransposeArgs t, int B) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ float tile[32][33];
  const int k0 = blockIdx.x * 32, b0 = blockIdx.y * 32, K = t.cols[blockIdx.z];
  const float* in = t.in[blockIdx.z];
  float* out = t.out[blockIdx.z];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (k0 >= K) return;
#pragma unroll
  for (int i = 0; i < 32; i += 8)
    if (b0 + y + i < B && k0 + x < K) tile[y + i][x] = in[(int64_t)(b0 + y + i) * K + k0 + x];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 32; i += 8)
    if (k0 + y + i < K && b0 + x < B) out[(int64_t)(k0 + y + i) * B + b0 + x] = tile[x][y + i];
}

template <int BH>
cudaError_t launch_step(const StepParams& p, cudaStream_t s) {
  auto kern = gru_step_kernel<BH>;
  constexpr size_t smem = step_smem<BH>();
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3((unsigned)(p.H / p.bh), (unsigned)((p.B + 31) / 32)), dim3(kStepWarps * 32), smem, s, p);
}

bool fused_step_supported(const grim_gru* g, int64_t B) {
  if (g->L > kStepMaxLayers || B > 65535 * 32) return false;
  for (int l = 0; l < g->L; ++l)
    if (!g->Wih[(size_t)l]->d_rc_head || !g->Whh[(size_t)l]->d_rc_head || g->Wih[(size_t)l]->bh != g->bh) return false;
  return true;
}

grim_status_t fused_step(grim_gru* g, const float* x, int64_t B, float* h, float* y, cudaStream_t s) {
  const int64_t H = g->H;
  TransposeArgs t = {};
  int widest = (int)g->Wih[0]->K;
  t.in[0] = x; t.out[0] = g->d_xT; t.cols[0] = widest;
  for (int l = 0; l < g->L; ++l) {
    t.in[l + 1] = h + (int64_t)l * B * H;
    t.out[l + 1] = g->d_gi[(size_t)l];  // H x B; the new state follows it (a layer's scratch holds at least 6 * H * B floats)
    t.cols[l + 1] = (int)H;
  }
  widest = std::max(widest, (int)H);
  cudaError_t e = launch_pdl(transpose_states_kernel, dim3((unsigned)((widest + 31) / 32), (unsigned)((B + 31) / 32), (unsigned)(g->L + 1)),
                             dim3(256), 0, s, t, (int)B);
  count_launch();
  for (int l = 0; l < g->L && e == cudaSuccess; ++l) {
    const grim_bcr* w[2] = {g->Wih[(size_t)l], g->Whh[(size_t)l]};
    StepParams p;
    for (int m = 0; m < 2; ++m) {
      p.w[m].head = w[m]->d_rc_head; p.w[m].blob = w[m]->d_rc_blob; p.w[m].nbc = (int)w[m]->nbc; p.w[m].bw = w[m]->bw;
      p.a[m].ncols = B; p.a[m].x_sk = B; p.a[m].x_sq = 1; p.a[m].x_dtype = GRIM_F32;
    }
    p.a[0].X = l == 0 ? g->d_xT : g->d_gi[(size_t)l - 1] + H * B;
    p.a[1].X = g->d_gi[(size_t)l];
    p.pos[0] = g->d_pos_of_band_ih[(size_t)l]; p.pos[1] = g->d_pos_of_band[(size_t)l];
    p.bias[0] = g->d_bih[(size_t)l]; p.bias[1] = g->d_bhh[(size_t)l];
    p.h = h + (int64_t)l * B * H;
    p.hT = l + 1 < g->L ? g->d_gi[(size_t)l] + H * B : nullptr;
    p.y = l + 1 == g->L ? y : nullptr;
    p.B = B; p.H = (int)H; p.bh = g->bh;
    // the eight warps of a gate are dealt to the two matrices by their block columns
    const double share = (double)w[0]->nbc / (double)(w[0]->nbc + w[1]->nbc);
    p.part[0] = std::min(7, std::max(1, (int)(8 * share + 0.5)));
    p.part[1] = 8 - p.part[0];
    e = g->bh <= 4 ? launch_step<4>(p, s) : (g->bh <= 8 ? launch_step<8>(p, s) : launch_step<16>(p, s));
    count_launch();
  }
  if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
  g->last_stream = s;
  return GRIM_OK;
}

// h'[b, u] = (1 - z) * n + z * h[b, u] with r, z, n from the two pre-activation buffers (batch-major, 3H per row);
// the state is updated in place and copied to y when given.
__global__ void gru_gate_kernel(const float* __restrict__ gi, const float* __restrict__ gh, float* __restrict__ h,
                                float* __restrict__ y, int64_t B, int64_t H) {
  const int64_t total = B * H;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i / H, u = i - b * H;
    const float* a = gi + b * 3 * H;
    const float* q = gh + b * 3 * H;
    const float r = sigmoidf_(a[u] + q[u]);
    const float z = sigmoidf_(a[H + u] + q[H + u]);
    const float n = tanhf(a[2 * H + u] + r * q[2 * H + u]);
    const float hn = (1.f - z) * n + z * h[i];
    h[i] = hn;
    if (y) y[i] = hn;
  }
}
}  // namespace

extern "C" grim_status_t grim_gru_step(grim_gru_t g, const float* x, int64_t B, float* h, float* y, grim_stream_t stream) {
  if (!g || !x || !h || B <= 0) return GRIM_ERR_INVALID_ARG;
  if (2 * B > g->max_T) return GRIM_ERR_SHAPE;  // both pre-activation buffers of a layer live in its T x 3H scratch
  cudaStream_t s = (cudaStream_t)stream;
  if (fused_step_supported(g, B)) return fused_step(g, x, B, h, y, s);
  const int64_t H = g->H;
  const float* in = x;
  for (int l = 0; l < g->L; ++l) {
    float* hl = h + (int64_t)l * B * H;
    float* gi = g->d_gi[(size_t)l];
    float* gh = gi + B * 3 * H;
    const grim_bcr* mats[2] = {g->Wih[(size_t)l], g->Whh[(size_t)l]};
    const float* rhs[2] = {in, hl};
    float* outs[2] = {gi, gh};
    const float* bias[2] = {g->d_bih[(size_t)l], g->d_bhh[(size_t)l]};
    for (int t = 0; t < 2; ++t) {
      // batch-major operands: X(k, b) at b * K + k, Y(r, b) at b * 3H + r
      SpmmArgs a;
      a.X = rhs[t]; a.Y = outs[t]; a.ncols = B;
      a.x_sk = 1; a.x_sq = mats[t]->K; a.y_sr = 1; a.y_sq = 3 * H;
      a.x_dtype = GRIM_F32; a.y_dtype = GRIM_F32;
      a.bias = bias[t];
      const grim_status_t st = launch_cuda_cores(mats[t], a, s);
      if (st != GRIM_OK) return st;
    }
    const int64_t total = B * H;
    gru_gate_kernel<<<(unsigned)std::min<int64_t>((total + 255) / 256, (int64_t)sm_count(g->device) * 8), 256, 0, s>>>(
        gi, gh, hl, l == g->L - 1 ? y : nullptr, B, H);
    count_launch();
    if (cudaGetLastError() != cudaSuccess) return GRIM_ERR_CUDA;
    in = hl;
  }
  g->last_stream = s;
  return GRIM_OK;
}
