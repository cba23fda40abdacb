// Direct CUDA-core kernel for Y = W * X and for convolutions (Sections 3.1, 4.4, 4.5): small and middle-sized products.
//
// A warp multiplies one row band with 32 * NC output columns, or, when that gives the GPU too few warps, a share of the
// band's block columns; the shares of a band sit in the same thread block and meet in shared memory, so there is no
// cleared output, no atomics and no second pass: one launch per product.  Everything is read straight from global
// memory (grim_rowwalk.cuh); activations that several bands need come from L1 or L2.
#include <algorithm>

#include "grim_internal.h"
#include "grim_rowwalk.cuh"

namespace grim {
namespace {

constexpr int kDWarps = 8;  // warps per thread block; 16 when sixteen of them share a band

struct DParams {
  RowWalk w;
  const uint32_t* band_order;
  int nbr, M, bh;
  int parts;  // warps that share a band: 1, 2, 4, 8 or 16
  SpmmArgs a;
};

// floats between two rows of a warp's partial sums: neighbouring rows four banks apart, so that reads down the rows
// (outputs stored column by column) are free of conflicts too
__host__ __device__ constexpr int part_ld(int nc) { return 32 * nc + 4; }
constexpr size_t direct_smem(int warps, int bh, int nc) { return (size_t)warps * ((size_t)bh * part_ld(nc) + kWalkBufFloats) * 4; }

template <int BH, int NC, int XV, typename XT, int CONV>
__global__ void __launch_bounds__(NC == 4 ? 256 : 512, NC == 4 ? 2 : 1) bcr_direct_kernel(const DParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(16) float dsm[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int nwarps = blockDim.x >> 5, bpc = nwarps / p.parts;  // bands of this thread block
  const int lb = warp / p.parts, part = warp - lb * p.parts;
  const int pos = blockIdx.y * bpc + lb;
  const SpmmArgs& a = p.a;
  const int64_t q0 = (int64_t)blockIdx.x * (32 * NC);
  constexpr int LD = part_ld(NC);
  float* wbuf = dsm + warp * kWalkBufFloats;
  float* sums = dsm + nwarps * kWalkBufFloats;  // [warp][row][column]

  float acc1[NC == 1 ? BH : 1];
  unsigned long long acc2[NC == 1 ? 1 : BH][NC == 1 ? 1 : NC / 2];
#pragma unroll
  for (int r = 0; r < BH; ++r) {
    if (NC == 1) acc1[NC == 1 ? r : 0] = 0.f;
#pragma unroll
    for (int c = 0; c < NC / 2; ++c) acc2[NC == 1 ? 0 : r][NC == 1 ? 0 : c] = 0ull;
  }
  // whatever earlier launches in the stream wrote is complete and visible after this; before it only the packed matrix
  // is touched
  auto wait_stream = [] { asm volatile("griddepcontrol.wait;" ::: "memory"); };
  if (pos < p.nbr) {
    WalkCols<NC, XV> wc;
    walk_setup<NC, XV, XT, CONV>(a, q0, lane, wc);
    // (one column per lane: the few columns that the lane-per-column kernels, which touch nothing but kept weights, took before)
    row_walk<BH, NC, XV, XT, CONV, NC == 1>(p.w, a, pos, part, p.parts, wc, wbuf, lane, acc1, acc2, wait_stream);
  } else {
    wait_stream();
  }
#pragma unroll
  for (int r = 0; r < BH; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c) sums[(warp * BH + r) * LD + walk_col<XV>(c, lane)] = walk_value<BH, NC>(acc1, acc2, r, c);
  __syncthreads();

  // the band's warps add the shares up, apply bias and activation and store
  if (pos >= p.nbr) return;
  const int64_t band = p.band_order[pos];
  const float* mine = sums + (size_t)lb * p.parts * BH * LD;
  const int64_t ohw = CONV ? (int64_t)a.OH * a.OW : 1;
  const bool down = !CONV && a.y_sq != 1;  // outputs stored column by column: rows run fastest
  for (int i = part * 32 + lane; i < BH * 32 * NC; i += 32 * p.parts) {
    const int r = down ? i % BH : i / (32 * NC), c = down ? i / BH : i % (32 * NC);
    const int64_t row = band * p.bh + r, q = q0 + c;
    if (r >= p.bh || row >= p.M || q >= a.ncols) continue;
    float t = 0.f;
    for (int s = 0; s < p.parts; ++s) t += mine[(s * BH + r) * LD + c];
    if (a.bias) t += __ldg(a.bias + row);
    if (a.relu) t = fmaxf(t, 0.f);
    int64_t off;
    if (CONV) {
      const int64_t img = q / ohw;
      off = (img * p.M + row) * ohw + (q - img * ohw);
    } else {
      off = row * a.y_sr + q * a.y_sq;
    }
    if (a.y_dtype == GRIM_F32) static_cast<float*>(a.Y)[off] = t;
    else static_cast<__nv_bfloat16*>(a.Y)[off] = __float2bfloat16_rn(t);
  }
}

template <int BH, int NC, int XV, typename XT, int CONV>
cudaError_t launch_one(const DParams& p, dim3 grid, cudaStream_t s) {
  auto kern = bcr_direct_kernel<BH, NC, XV, XT, CONV>;
  const int warps = std::max(p.parts, kDWarps);
  const size_t smem = direct_smem(warps, BH, NC);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, grid, dim3(32 * warps), smem, s, p);
}

template <int BH>
cudaError_t launch_rows(const DParams& p, int nc, int xv, dim3 grid, cudaStream_t s) {
  if (p.a.x_dtype == GRIM_BF16) {
    if (p.a.conv) return nc == 4 ? launch_one<BH, 4, 1, __nv_bfloat16, 1>(p, grid, s) : launch_one<BH, 2, 1, __nv_bfloat16, 1>(p, grid, s);
    return nc == 4 ? launch_one<BH, 4, 1, __nv_bfloat16, 0>(p, grid, s)
                   : (nc == 2 ? launch_one<BH, 2, 1, __nv_bfloat16, 0>(p, grid, s) : launch_one<BH, 1, 1, __nv_bfloat16, 0>(p, grid, s));
  }
  if (p.a.conv) return nc == 4 ? launch_one<BH, 4, 1, float, 1>(p, grid, s) : launch_one<BH, 2, 1, float, 1>(p, grid, s);
  if (nc == 4) return xv == 4 ? launch_one<BH, 4, 4, float, 0>(p, grid, s) : launch_one<BH, 4, 1, float, 0>(p, grid, s);
  if (nc == 2) return xv == 2 ? launch_one<BH, 2, 2, float, 0>(p, grid, s) : launch_one<BH, 2, 1, float, 0>(p, grid, s);
  return launch_one<BH, 1, 1, float, 0>(p, grid, s);
}

}  // namespace

// 32, or 32 + columns per lane + 256 * warps per band
bool direct_choice(int tile_n) {
  if (tile_n == 32) return true;
  const int nc = tile_n % 256 - 32, parts = tile_n / 256;
  return tile_n > 0 && (nc == 1 || nc == 2 || nc == 4) && (parts == 1 || parts == 2 || parts == 4 || parts == 8 || (parts == 16 && nc < 4));
}

bool direct_path_supported(const grim_bcr* h, const SpmmArgs& a) {
  if (h->device < 0 || !h->d_rc_head) return false;
  if (a.ncols <= 0 || a.ncols > (int64_t(1) << 31) - 256) return false;
  if ((h->nbr + kDWarps - 1) / kDWarps > 65535) return false;  // bands are dealt to the grid's second dimension
  if (!a.conv && a.x_sk * (a.x_dtype == GRIM_F32 ? 4 : 2) >= (int64_t(1) << 32)) return false;
  if (a.conv && (a.KH > 16 || a.KW > 16 || (int64_t)a.C * a.H * a.W >= (int64_t(1) << 31))) return false;
  return true;
}

double direct_time(const grim_bcr* h, const SpmmArgs& a) {
  const bool few = a.ncols <= 64;
  const double per_chunk = h->bh <= 4 ? (few ? 0.29e-3 : 0.33e-3) : (h->bh <= 8 ? (few ? 0.44e-3 : 0.5e-3) : (few ? 0.6e-3 : 1.0e-3));
  return 4.0 + per_chunk * (double)h->rc_chunks * (double)((a.ncols + 127) / 128);
}

// Where the direct kernel is the faster of the CUDA-core kernels (measured on square matrices of 512 to 8192, pruning rate
// 8, the three block shapes; times in us, slab kernel -> direct kernel).
bool direct_preferred(const grim_bcr* h, const SpmmArgs& a) {
  if (!direct_path_supported(h, a)) return false;
  const double flops = 2.0 * (double)h->nnz * (double)a.ncols;
  // Convolutions: the slab kernel's gather costs more than it saves at every size (512 channels, 28 x 28: one image
  // 86 -> 63, 32 images 1320 -> 1220; 64 channels, 112 x 112: 58 -> 26; 5 x 5 on 96 channels, 17 x 23: 416 -> 18).
  if (a.conv) return true;
  if (a.ncols <= kSkinnyMaxN) {
    // Few columns leave most lanes idle, so the time goes with the number of chunks (about 2.5 us and 0.3 ns each).  Against
    // the gathering kernel, which has more to set up: up to some 5000 chunks (1024^2, 8 x 32, N = 7: 3.4 against 5.2; 512^2:
    // 3.0 against 5.2), and where that one needs two passes up to 17000 (2048^2, 16 x 64, N = 16: 6.7 against 7.6).
    // Handles that hold only the wide regime's layouts go on refusing what grim.h says they refuse: they only take these widths
    // from eight columns on, and where the tensor-core tile or the slab kernel's narrow tile is there for them.
    if ((h->flags & GRIM_PACK_WIDE_ONLY) && h->gemv_ok &&
        (a.ncols < 8 || !(h->dtype == GRIM_F32 ? h->bh >= 8 && ffma_path_supported(h, a) : tc_path_supported(h, a) && h->tc_mtiles >= 8)))
      return false;
    if (a.x_dtype == GRIM_BF16 && a.ncols >= 8) return !h->d_chunks && h->rc_chunks <= 5000;
    return h->rc_chunks <= (h->bh > 8 && a.ncols > 8 ? 17000 : 5000) && a.ncols >= 5;
  }
  // The slab kernel needs rows of X that TMA can fetch; its other loaders are slow (N = 1023: 1477 -> 1213, N = 131 in
  // bf16: 328 -> 30), except that a slab row of 16-row bands is used often enough to pay for them in large products.
  if (!slab_rows_by_tma(a)) return a.x_dtype == GRIM_BF16 || h->bh <= 8 || flops <= 1e9;
  // Otherwise: whichever is estimated to be done first.  The direct kernel's time goes with the chunks and 128-column tiles
  // (0.33, 0.5 and 1.0 ns each for 4, 8 and 16 rows, less for up to 64 columns), the slab kernel's with the stages it takes one after the other.
  // (1024^2, N = 128: 6.4 against 11; 2048^2, 4 x 16, N = 256: 44 against 26; 8 x 32: 23 against 22; 4096 x 1024, N = 256:
  // 26 against 21; 1024 x 4096: 22 against 33.)
  return direct_time(h, a) <= slab_time(h, a);
}

grim_status_t launch_direct(const grim_bcr* h, const SpmmArgs& a, cudaStream_t s) {
  if (!direct_path_supported(h, a)) return GRIM_ERR_UNSUPPORTED;
  DParams p;
  p.w.head = h->d_rc_head; p.w.blob = h->d_rc_blob; p.w.nbc = (int)h->nbc; p.w.bw = h->bw;
  p.band_order = h->d_band_order; p.nbr = (int)h->nbr; p.M = (int)h->M; p.bh = h->bh;
  p.a = a;
  const int BHc = h->bh <= 4 ? 4 : (h->bh <= 8 ? 8 : 16);
  const int sms = sm_count(h->device);
  int nc, parts;
  if (a.tile_n > 32 && direct_choice(a.tile_n)) {
    nc = a.tile_n % 32; parts = a.tile_n / 256;
  } else {
    auto warps = [&](int n) { return ((a.ncols + 32 * n - 1) / (32 * n)) * h->nbr; };
    nc = a.ncols <= 32 && !a.conv ? 1 : 2;
    if (a.ncols > 64 && warps(4) >= sms && 4 * ((a.ncols + 127) / 128) * 4 <= 5 * 2 * ((a.ncols + 63) / 64)) nc = 4;
    parts = 1;
    while (parts < (nc == 4 ? 8 : 16) && warps(nc) * parts * 2 <= (int64_t)sms * 16 && h->nbc >= 2 * parts) parts *= 2;
  }
  p.parts = parts;
  int xv = 1;
  if (!a.conv && a.x_dtype == GRIM_F32 && a.x_sq == 1 && nc > 1 && a.ncols % nc == 0 && a.x_sk % nc == 0 &&
      reinterpret_cast<uintptr_t>(a.X) % (4 * nc) == 0)
    xv = nc;
  const int64_t gx = (a.ncols + 32 * nc - 1) / (32 * nc), bpc = std::max(kDWarps, parts) / parts, gy = (h->nbr + bpc - 1) / bpc;
  if (gy > 65535) return GRIM_ERR_UNSUPPORTED;
  dim3 grid((unsigned)gx, (unsigned)gy);
  const cudaError_t e = BHc == 4 ? launch_rows<4>(p, nc, xv, grid, s) : (BHc == 8 ? launch_rows<8>(p, nc, xv, grid, s) : launch_rows<16>(p, nc, xv, grid, s));
  count_launch();
  if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
  return GRIM_OK;
}

}  // namespace grim
