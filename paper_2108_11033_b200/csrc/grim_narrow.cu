// Gathering kernel for 2 <= N <= 16 right-hand sides (Sections 3.1, 4.3, 4.4), on the chunk layout of the matrix-vector
// kernel: a chunk is up to 32 kept columns of one band with the same number of kept rows; lane l owns column l.
//
// A warp walks every `parts`-th chunk of one band.  Per chunk it copies the values (contiguous) and, for each of the 32
// columns, the row of X that the column meets into a small ring of its own in shared memory with asynchronous copies, three
// or four chunks ahead of the multiply; the column words run one further chunk ahead.  So nothing is shared between warps
// before the end, X is read straight from L2 whatever its size, and the shares of a band meet in shared memory: one launch,
// no cleared output, no atomics.  (The kernel it replaces staged X slice by slice for a whole thread block: 45 us for
// 3001 x 5003 at rate 8 in 4 x 16 blocks with N = 7, most of it waiting for the slices.)
//
// fp32: a lane holds one column's NQ activations and walks the rows of the band with packed two-column FMAs; the lanes'
// sums meet in a halving exchange at the end.
// bf16: the tensor core multiplies 16 kept columns at a time with mma.sync (m = columns of X, n = rows of the band, k =
// kept columns): the gathered rows of X are the transposed operand as ldmatrix delivers it, the values are picked from the
// chunk with the columns' row masks.  (These products are bound by latency and by the gather, not by multiply rate: a
// tcgen05 tile would be 128 x 16 with a k step per kept column of any band, i.e. dense.)
#include <cuda_bf16.h>

#include <algorithm>

#include "grim_device.cuh"
#include "grim_internal.h"

namespace grim {
namespace {

constexpr int kNWarps = 8;

struct NParams {
  const uint32_t* band_ptr;
  const ChunkDesc* chunks;
  const uint32_t* colwords;
  const uint8_t* vals;
  const uint32_t* band_order;
  const void* X;
  void* Y;
  int64_t ldx, ldy;
  int N, nbr, M, bh, y_dtype, parts;
};

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Shape of one ring stage of a warp: 32 column words, the values (and what lies between a 16-byte boundary and them), X rows.
template <int BH, int NQ, typename VT>
struct Stage {
  static constexpr int kRow = NQ * (int)sizeof(VT);       // bytes of a gathered row: 16, 32 or 64
  static constexpr int kVals = 128, kX = kVals + 32 * BH * (int)sizeof(VT) + 32;
  static constexpr int kBytes = kX + 32 * kRow;
  static constexpr int kDepth = BH * (int)sizeof(VT) >= 64 ? 3 : 4;
  // 16-byte piece p of row r: rows that eight lanes read together spread over all banks
  static __device__ __forceinline__ uint32_t piece(int r, int p) { return (uint32_t)(kX + r * kRow + ((p ^ (kRow == 64 ? (r >> 1) & 3 : (kRow == 32 ? (r >> 2) & 1 : 0))) << 4)); }
};

template <int BH, int NQ, typename VT>
__host__ __device__ constexpr size_t narrow_smem() {
  return (size_t)kNWarps * Stage<BH, NQ, VT>::kDepth * Stage<BH, NQ, VT>::kBytes;
}

__device__ __forceinline__ void nfma2(unsigned long long& acc, unsigned long long w2, unsigned long long x2) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(w2), "l"(x2));
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// A warp's sums, product by kept product: what the tensor core's cannot be used for when activations are not finite, because it
// multiplies the rows of a band that do not keep a column by zero.  Lane l works out outputs l, l + 32, ...
template <int BH, int NQ>
__device__ __noinline__ void kept_products(const NParams& p, int pos, int part, int q0, int lane, float* mine) {
  const unsigned short* vals = reinterpret_cast<const unsigned short*>(p.vals);
  const unsigned short* X = static_cast<const unsigned short*>(p.X);
  const int c0 = pos < p.nbr ? (int)__ldg(p.band_ptr + pos) + part : 0, c1 = pos < p.nbr ? (int)__ldg(p.band_ptr + pos + 1) : 0;
  for (int i = lane; i < BH * NQ; i += 32) {
    const int r = i / NQ, q = q0 + i % NQ;
    float t = 0.f;
    for (int c = c0; c < c1 && q < p.N; c += p.parts) {
      const ChunkDesc d = p.chunks[c];
      const uint32_t ncols = d.ncols_kr & 0xFFFFu;
      for (uint32_t j = 0; j < ncols; ++j) {
        const uint32_t w = __ldg(p.colwords + (size_t)c * 32 + j), rm = w >> 16;
        if (!((rm >> r) & 1u)) continue;
        const uint32_t v = vals[d.val_off + (uint32_t)__popc(rm & ((1u << r) - 1u)) * ncols + j];
        const uint32_t x = X[(int64_t)(w & 0xFFFFu) * p.ldx + q];
        t = fmaf(__uint_as_float(v << 16), __uint_as_float(x << 16), t);
      }
    }
    mine[i] = t;
  }
}

// Blocks per SM: as many as registers allow.  In bf16 four, and their rings have to leave room for it (the sums take the place of
// the rings): with three, products of some four thousand warps take a second round (4096^2, 8 x 32 at rate 8, N = 16: 10.3 -> 8.8 us).
template <int BH, int NQ, typename VT>
__global__ void __launch_bounds__(kNWarps * 32, sizeof(VT) == 2 ? 4 : (BH * NQ >= 128 ? 1 : 2)) bcr_narrow_kernel(const __grid_constant__ NParams p) {
  using S = Stage<BH, NQ, VT>;
  constexpr bool MMA = sizeof(VT) == 2;
  constexpr int D = S::kDepth;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(16) uint8_t nsm[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int lb = warp / p.parts, part = warp - lb * p.parts, bpc = kNWarps / p.parts;
  const int pos = blockIdx.x * bpc + lb;
  const int q0 = blockIdx.y * NQ;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(nsm) + (uint32_t)warp * (D * S::kBytes);
  const uint8_t* ring_p = nsm + (size_t)warp * (D * S::kBytes);
  constexpr int kSumsLd = D * S::kBytes / 4;  // a warp's sums, [row][column], take the place of its ring
  static_assert(D * S::kBytes >= BH * NQ * 4, "sums fit the ring");
  float* sums = reinterpret_cast<float*>(nsm);

  int c = 0, end = 0;  // next chunk of this warp to be fetched
  if (pos < p.nbr) {
    end = (int)__ldg(p.band_ptr + pos + 1);
    c = (int)__ldg(p.band_ptr + pos) + part;
  }
  const int n_chunks = c < end ? (end - c + p.parts - 1) / p.parts : 0;

  struct Head { uint32_t val_off, ncols_kr, word; };
  auto load_head = [&]() {
    Head h{0u, 0u, 0u};
    if (c < end) {
      h.val_off = __ldg(&p.chunks[c].val_off);
      h.ncols_kr = __ldg(&p.chunks[c].ncols_kr);
      h.word = __ldg(p.colwords + (size_t)c * 32 + lane);  // words past the last column are 0: no row kept
      c += p.parts;
    }
    return h;
  };
  auto fetch = [&](const Head& h, int slot) {
    if (h.ncols_kr) {
      const uint32_t st = ring + (uint32_t)slot * S::kBytes;
      asm volatile("st.shared.u32 [%0], %1;" ::"r"(st + (uint32_t)lane * 4u), "r"(h.word) : "memory");
      const uint64_t a0 = (uint64_t)h.val_off * sizeof(VT), al = a0 & ~(uint64_t)15;
      const uint32_t bytes = (uint32_t)(a0 - al) + (h.ncols_kr & 0xFFFFu) * (h.ncols_kr >> 16) * (uint32_t)sizeof(VT);
      for (uint32_t i = (uint32_t)lane * 16u; i < bytes; i += 512u) cp16(st + S::kVals + i, p.vals + al + i, true);
      const VT* X = static_cast<const VT*>(p.X) + q0;
      constexpr int PPR = S::kRow / 16, EP = 16 / (int)sizeof(VT);  // pieces per row, elements per piece
#pragma unroll
      for (int i = 0; i < PPR; ++i) {
        const int r = i * (32 / PPR) + lane / PPR, pc = lane % PPR;
        const uint32_t w = __shfl_sync(0xffffffffu, h.word, r);
        cp16(st + S::piece(r, pc), X + (int64_t)(w & 0xFFFFu) * p.ldx + pc * EP, (w >> 16) && q0 + pc * EP < p.N);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // accumulators: fp32: [row][pair of columns]; bf16: fragments of 16 x 8 (columns of X x rows of the band)
  constexpr int NP = NQ / 2, NT = BH == 16 ? 2 : 1;
  unsigned long long acc[MMA ? 1 : BH][MMA ? 1 : NP];
  float frag[NT][4];
#pragma unroll
  for (int r = 0; r < (MMA ? 1 : BH); ++r)
#pragma unroll
    for (int q = 0; q < (MMA ? 1 : NP); ++q) acc[r][q] = 0ull;
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) frag[t][i] = 0.f;

  {
    Head first[D];
#pragma unroll
    for (int d = 0; d < D; ++d) first[d] = load_head();
    // whatever earlier launches in the stream wrote is complete and visible after this; before it only the packed matrix
    // is touched
    asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
    for (int d = 0; d < D; ++d) fetch(first[d], d);
  }
  Head ahead = load_head();
  int slot = 0;
  // (the head of the chunk that is multiplied is not kept: its words are in the stage, its shape is reloaded from L1)
  int cur = pos < p.nbr ? (int)__ldg(p.band_ptr + pos) + part : 0;
  for (int n = 0; n < n_chunks; ++n, cur += p.parts) {
    const uint32_t val_off = __ldg(&p.chunks[cur].val_off);
    const uint32_t ncols = __ldg(&p.chunks[cur].ncols_kr) & 0xFFFFu;
    cp_wait<D - 1>();
    __syncwarp();
    const uint8_t* st = ring_p + (size_t)slot * S::kBytes;
    const uint32_t st_s = ring + (uint32_t)slot * S::kBytes;
    const VT* v0 = reinterpret_cast<const VT*>(st + S::kVals + (((uint64_t)val_off * sizeof(VT)) & 15));
    if constexpr (!MMA) {
      const uint32_t rm = reinterpret_cast<const uint32_t*>(st)[lane] >> 16;
      ulonglong2 x[NQ / 4];
#pragma unroll
      for (int i = 0; i < NQ / 4; ++i) x[i] = *reinterpret_cast<const ulonglong2*>(st + S::piece(lane, i));
      const float* at = reinterpret_cast<const float*>(v0) + lane;
#pragma unroll
      for (int r = 0; r < BH; ++r) {
        if ((rm >> r) & 1u) {
          const float w = *at;
          at += ncols;
          unsigned long long w2;
          asm("mov.b64 %0, {%1, %1};" : "=l"(w2) : "f"(w));
#pragma unroll
          for (int i = 0; i < NQ / 4; ++i) {
            nfma2(acc[MMA ? 0 : r][MMA ? 0 : 2 * i], w2, x[i].x);
            nfma2(acc[MMA ? 0 : r][MMA ? 0 : 2 * i + 1], w2, x[i].y);
          }
        }
      }
    } else {
      const uint32_t* words = reinterpret_cast<const uint32_t*>(st);
      const unsigned short* vv = reinterpret_cast<const unsigned short*>(v0);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h == 1 && ncols <= 16) break;  // (uniform)
        uint32_t a0, a1 = 0u, a2, a3 = 0u;
        if (NQ == 16) {
          const uint32_t at = st_s + S::piece(16 * h + (lane & 7) + 8 * (lane >> 4), (lane >> 3) & 1);
          asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3) : "r"(at) : "memory");
        } else {
          const uint32_t at = st_s + S::piece(16 * h + (lane & 15), 0);
          asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(a0), "=r"(a2) : "r"(at) : "memory");
        }
        const int j0 = 16 * h + 2 * (lane & 3);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const int row = (lane >> 2) + 8 * t;  // rows from BH on are in no mask
          uint32_t b[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int j = j0 + (i & 1) + 8 * (i >> 1);
            const uint32_t rm = words[j] >> 16;
            b[i] = 0u;
            if ((rm >> row) & 1u) b[i] = vv[(uint32_t)__popc(rm & ((1u << row) - 1u)) * ncols + (uint32_t)j];
          }
          mma16816(frag[t], a0, a1, a2, a3, b[0] | b[1] << 16, b[2] | b[3] << 16);
        }
      }
    }
    __syncwarp();  // every lane is done with the stage before it is filled again
    fetch(ahead, slot);
    ahead = load_head();
    if (++slot == D) slot = 0;
  }
  cp_wait<0>();

  __syncwarp();
  float* mine = sums + warp * kSumsLd;
  if constexpr (!MMA) {
    const int row = warp_row<BH>(lane);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      float t[BH];
#pragma unroll
      for (int r = 0; r < BH; ++r) {
        const unsigned long long v = acc[MMA ? 0 : r][MMA ? 0 : q / 2];
        t[r] = __uint_as_float((unsigned)((q & 1) ? v >> 32 : v));
      }
      warp_reduce_rows<BH>(t, lane);
      mine[row * NQ + q] = t[0];  // lanes that share a row hold the same total
    }
  } else {
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int m = (lane >> 2) + 8 * (i >> 1), n = 2 * (lane & 3) + (i & 1) + 8 * t;
        if (m < NQ && n < BH) mine[n * NQ + m] = frag[t][i];
      }
    // an infinity or a NaN among the activations has reached every row of the band: those sums are not finite
    bool finite = true;
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int i = 0; i < 4; ++i) finite = finite && fabsf(frag[t][i]) <= 3.4028234e38f;
    if (!__all_sync(0xffffffffu, finite)) {
      __syncwarp();
      kept_products<BH, NQ>(p, pos, part, q0, lane, mine);
    }
  }
  __syncthreads();
  for (int i = tid; i < bpc * BH * NQ; i += kNWarps * 32) {
    const int b = i / (BH * NQ), rq = i - b * (BH * NQ), r = rq / NQ, q = q0 + rq % NQ;
    const int at = blockIdx.x * bpc + b;
    if (at >= p.nbr || r >= p.bh || q >= p.N) continue;
    const int64_t row = (int64_t)__ldg(p.band_order + at) * p.bh + r;
    if (row >= p.M) continue;
    float t = 0.f;
    for (int s = 0; s < p.parts; ++s) t += sums[(b * p.parts + s) * kSumsLd + rq];
    if (p.y_dtype == GRIM_F32) static_cast<float*>(p.Y)[row * p.ldy + q] = t;
    else static_cast<__nv_bfloat16*>(p.Y)[row * p.ldy + q] = __float2bfloat16_rn(t);
  }
}

template <int BH, int NQ, typename VT>
cudaError_t launch_one(const NParams& p, int sms, cudaStream_t s) {
  auto kern = bcr_narrow_kernel<BH, NQ, VT>;
  constexpr size_t smem = narrow_smem<BH, NQ, VT>();
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  const int bpc = kNWarps / p.parts;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((p.nbr + bpc - 1) / bpc), (unsigned)((p.N + NQ - 1) / NQ));
  cfg.blockDim = dim3(kNWarps * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  // No more shared memory than the blocks of this launch take: what is left is L1, where the gathered rows of X come from (as many
  // blocks as fit leave 12 KB; bf16, rate 4, N = 16, two blocks to an SM: 4096^2, 16 x 64: 13.4 -> 10.3 us; 2048 x 8192, 8 x 32: 19.8 -> 13.5).
  const int64_t per_sm = ((int64_t)cfg.gridDim.x * cfg.gridDim.y + sms - 1) / sms;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = (unsigned)std::min<int64_t>(100, (per_sm * (int64_t)(smem + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024));
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p);
}
template <int BH>
cudaError_t launch_rows(const NParams& p, bool bf16, int sms, cudaStream_t s) {
  if (bf16) return p.N <= 8 ? launch_one<BH, 8, __nv_bfloat16>(p, sms, s) : launch_one<BH, 16, __nv_bfloat16>(p, sms, s);
  if (p.N <= 4) return launch_one<BH, 4, float>(p, sms, s);
  if (BH <= 8 && p.N > 8) return launch_one<(BH <= 8 ? BH : 8), 16, float>(p, sms, s);
  return launch_one<BH, 8, float>(p, sms, s);  // (16 x 16 accumulators do not fit: two passes of eight columns)
}

// Rows of X whose 16-byte pieces are not all aligned are copied into the handle's scratch first, padded with zeros to
// whole pieces: a gather element by element costs more than this pass (3001 x 5003, N = 7: 22.8 us without it).
template <typename T>
__global__ void __launch_bounds__(256) pad_rows_kernel(const T* __restrict__ X, int64_t ldx, int K, int N, int np, uint4* __restrict__ out) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int i = blockIdx.x * 256 + threadIdx.x, k = i / np, pc = i - k * np;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (k >= K) return;
  constexpr int E = 16 / (int)sizeof(T);
  union { uint4 v; T e[E]; } u;
  u.v = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (pc * E + e < N) u.e[e] = X[(int64_t)k * ldx + pc * E + e];
  out[i] = u.v;
}

}  // namespace

// Where this kernel is the best of those that take 2 <= N <= 16 (measured on square matrices of 512 to 8192 at rate 8 in the
// three block shapes, both types, N = 2, 4, 7, 8, 16; times in us).
bool narrow_preferred(const grim_bcr* h, const SpmmArgs& a) {
  const int64_t N = a.ncols;
  if (!narrow_path_supported(h, N)) return false;
  // up to four columns and eight rows to a band the streaming kernel's larger transfers win (8192^2, 8 x 32, N = 4: 17.5
  // against 21.5; bf16 19.8 against 21); with 16 rows its lanes walk mostly pruned rows (16 x 64: 29 against 19)
  if (N <= 4) return h->bh > 8;
  // The slab kernel's narrow tile, where it can fetch the rows and is estimated to be done first: against two passes over the
  // weights for 16 x 16 accumulators (5696^2, N = 16: 28 against 46; 640 x 5952: 21 against 8.6), and for more than eight columns
  // where many columns of W are kept in few rows each, because a gathered row of X costs the same whatever its column keeps
  // (8 x 32: 5376^2, heavy-tailed, N = 12: 37 against 50; 4096^2, uniform, N = 16: 20 against 15)
  if (h->dtype == GRIM_F32 && h->bh >= 8 && N > 8) return narrow_time(h) <= slab_time(h, a);
  return true;
}

double narrow_time(const grim_bcr* h) {
  return h->bh > 8 ? 4.0 + 11e-6 * (double)h->nnz + 9e-3 * (double)h->nbr : 1.0 + 1.05e-3 * (double)h->nchunks;
}

bool narrow_path_supported(const grim_bcr* h, int64_t N) {
  return h->device >= 0 && h->gemv_ok && h->d_chunks && N >= 2 && N <= kSkinnyMaxN && h->nbr < (int64_t(1) << 30);
}

grim_status_t launch_narrow(const grim_bcr* h, const void* X, int x_dtype, int64_t ldx, int64_t N, void* Y, int y_dtype, int64_t ldy,
                            int parts, cudaStream_t s) {
  if (x_dtype != h->dtype) return GRIM_ERR_DTYPE;
  if (!narrow_path_supported(h, N)) return GRIM_ERR_UNSUPPORTED;
  NParams p;
  p.band_ptr = h->d_gemv_band_ptr; p.chunks = h->d_chunks; p.colwords = h->d_colwords; p.vals = static_cast<const uint8_t*>(h->d_gemv_vals);
  p.band_order = h->d_band_order; p.X = X; p.Y = Y; p.ldx = ldx; p.ldy = ldy;
  p.N = (int)N; p.nbr = (int)h->nbr; p.M = (int)h->M; p.bh = h->bh; p.y_dtype = y_dtype;
  const int esz = x_dtype == GRIM_F32 ? 4 : 2;
  if ((N * esz) % 16 != 0 || (ldx * esz) % 16 != 0 || reinterpret_cast<uintptr_t>(X) % 16 != 0) {
    const int np = (int)((N * esz + 15) / 16), total = (int)h->K * np;
    uint4* pad = static_cast<uint4*>(h->d_xpad);
    const dim3 grid((unsigned)((total + 255) / 256));
    const cudaError_t e = esz == 4 ? launch_pdl(pad_rows_kernel<float>, grid, dim3(256), 0, s, static_cast<const float*>(X), ldx, (int)h->K, (int)N, np, pad)
                                   : launch_pdl(pad_rows_kernel<unsigned short>, grid, dim3(256), 0, s, static_cast<const unsigned short*>(X), ldx, (int)h->K, (int)N, np, pad);
    count_launch();
    if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
    p.X = pad;
    p.ldx = np * 16 / esz;
  }
  if (parts == 0) {
    // as many warps as hide the latency of the gathers without repeating a warp's fixed cost too often, and a few chunks
    // for each (8192 x 8192, 8 x 32: N = 16 in bf16 31 / 26 / 23 us with 2048 / 4096 / 8192 warps; N = 8 in fp32, whose warps
    // need twice the registers, 27.4 / 29.3 / 32.3; N = 16 in fp32, one block per SM, 49 / 53 / 55)
    const bool big = esz == 4 && (h->bh > 8 ? N > 4 : h->bh > 4 && N > 8);
    const int per_sm = esz == 2 || N <= 4 ? 64 : (big ? 8 : 16);
    parts = 1;
    const int64_t per_band = h->nchunks / h->nbr;
    while (parts < kNWarps && h->nbr * parts * 2 <= (int64_t)sm_count(h->device) * per_sm && per_band >= 2 * parts) parts *= 2;
  }
  p.parts = parts;
  const bool bf16 = x_dtype == GRIM_BF16;
  const int sms = sm_count(h->device);
  const cudaError_t e = h->bh <= 4 ? launch_rows<4>(p, bf16, sms, s) : (h->bh <= 8 ? launch_rows<8>(p, bf16, sms, s) : launch_rows<16>(p, bf16, sms, s));
  count_launch();
  if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
  return GRIM_OK;
}

}  // namespace grim
