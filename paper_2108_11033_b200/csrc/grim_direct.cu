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

namespace {
// Columns per lane and warps per band: enough warps to hide latency (some 16 per SM), four columns where that does not leave too
// much of the last tile unused.
struct Shape { int nc, parts; };
Shape shape_for(const grim_bcr* h, const SpmmArgs& a) {
  const int sms = sm_count(h->device);
  auto warps = [&](int n) { return ((a.ncols + 32 * n - 1) / (32 * n)) * h->nbr; };
  Shape s{a.ncols <= 32 && !a.conv ? 1 : 2, 1};
  if (a.ncols > 64 && warps(4) >= sms && 4 * ((a.ncols + 127) / 128) * 4 <= 5 * 2 * ((a.ncols + 63) / 64)) s.nc = 4;
  while (s.parts < (s.nc == 4 ? 8 : 16) && warps(s.nc) * s.parts * 2 <= (int64_t)sms * 16 && h->nbc >= 2 * s.parts) s.parts *= 2;
  return s;
}
}  // namespace

int direct_parts(const grim_bcr* h, const SpmmArgs& a) { return shape_for(h, a).parts; }

// What a warp does one after the other (its chunks), what all warps issue (chunks and bands times tiles).  Fitted to 400 products and
// 340 convolutions of 100 .. 8192 rows, 200 .. 8192 columns of W, N of 2 to 1024, rates 4 to 16: nine in ten within 15 %.
double direct_time(const grim_bcr* h, const SpmmArgs& a) {
  const Shape s = shape_for(h, a);
  const int b = h->bh <= 4 ? 0 : (h->bh <= 8 ? 1 : 2);
  const double tiles = (double)((a.ncols + 32 * s.nc - 1) / (32 * s.nc)) * s.nc;  // of 32 columns
  const double serial = (double)h->rc_chunks / ((double)h->nbr * s.parts), chunks = (double)h->rc_chunks * tiles * 1e-3, bands = (double)h->nbr * tiles * 1e-3;
  if (a.conv) {
    static const double c[2][3][4] = {{{2.3, 0.47, 0.10, 1.0}, {2.6, 0.95, 0.14, 1.8}, {3.3, 1.9, 0.09, 4.4}},     // fp32
                                      {{2.2, 0.59, 0.16, 1.0}, {3.1, 0.92, 0.30, 1.8}, {4.1, 1.9, 0.23, 4.4}}};   // bf16
    const double* v = c[a.x_dtype == GRIM_BF16][b];
    return v[0] + v[1] * serial + v[2] * chunks + v[3] * bands;
  }
  static const double c[2][3][4] = {{{1.8, 0.62, 0.06, 1.3}, {1.7, 0.86, 0.02, 2.8}, {2.5, 1.04, 0.02, 6.5}},      // N <= 64
                                    {{1.95, 0.41, 0.06, 0.4}, {2.25, 0.66, 0.06, 1.3}, {3.0, 1.04, 0.08, 5.0}}};  // wider
  const double* v = c[a.ncols > 64][b];
  return v[0] + v[1] * serial + v[2] * chunks + v[3] * bands;
}

// Where the direct kernel is the faster of the CUDA-core kernels.
bool direct_preferred(const grim_bcr* h, const SpmmArgs& a) {
  if (!direct_path_supported(h, a)) return false;
  // Convolutions: the slab kernel's gather costs more than it saves at every size (512 channels, 28 x 28: one image
  // 86 -> 63, 32 images 1320 -> 1220; 64 channels, 112 x 112: 58 -> 26; 5 x 5 on 96 channels, 17 x 23: 416 -> 18).
  if (a.conv) return true;
  if (a.ncols <= kSkinnyMaxN) {
    // Few columns leave most lanes idle and the chunks of a warp are walked one after the other; the gathering kernel has more to
    // set up (about 4 us) but takes 32 columns of W at a time, and where it needs two passes some 11 us per million weights
    // (1024^2, 8 x 32, N = 7: 3.4 against 5.2; 4032^2 at rate 16, 16 x 64, N = 14: 11.8 against 16.8; 640 x 5952, N = 16: 15.9
    // against 8.6; 256 x 8128, N = 11: 37.7 against 17.5).
    // Handles that hold only the wide regime's layouts go on refusing what grim.h says they refuse: they only take these widths
    // from eight columns on, and where the tensor-core tile or the slab kernel's narrow tile is there for them.
    if ((h->flags & GRIM_PACK_WIDE_ONLY) && h->gemv_ok &&
        (a.ncols < 8 || !(h->dtype == GRIM_F32 ? h->bh >= 8 && ffma_path_supported(h, a) : tc_path_supported(h, a) && h->tc_mtiles >= 8)))
      return false;
    if (a.ncols < 5 || (a.x_dtype == GRIM_BF16 && a.ncols >= 8 && h->d_chunks)) return false;
    // (fp32, 16-row blocks, more than eight columns: whatever takes them otherwise needs longer)
    const double other = h->dtype == GRIM_F32 && h->bh > 8 && a.ncols > 8 ? std::min(narrow_time(h), slab_time(h, a)) : 0.0;
    return direct_time(h, a) <= std::max(5.0, 1.1 * other);
  }
  // bf16: the slab kernel widens what it gathers, element by element, where TMA cannot fetch the rows (N = 131: 328 -> 30)
  if (a.x_dtype == GRIM_BF16 && !slab_rows_by_tma(a)) return true;
  // X stored column by column (the GRU's inputs where they are not turned around): a lane's loads do not coalesce, so wide ones are
  // better gathered (GRU step of a batch of 64, 4 x 16: 184 against 155; 48: equal; 32: 84 against 150; 8 x 32: 99 against 172 at
  // 64; a sequence of 400 steps 1320 against 1297)
  if (a.x_sq != 1) return a.ncols <= (h->bh <= 4 ? 48 : 384) && (h->bh <= 8 || 2.0 * (double)h->nnz * (double)a.ncols <= 1e9);
  // Otherwise: whichever is estimated to be done first.  The slab kernel's time goes with the stages it takes one after the other
  // (slab against direct: 1024^2, N = 128: 11 - 6.4; 2048^2, 4 x 16, N = 256: 26 - 42; N = 131: 59 - 82; 4096^2, 8 x 32, N = 64: 36 -
  // 32; 8192^2, 4 x 16, N = 32: 347 - 420; 1664 x 896, 16 x 64, N = 1000: 28 - 46).
  // The estimate of the gathering loader is the less certain one.
  return direct_time(h, a) <= slab_time(h, a) * (slab_rows_by_tma(a) ? 1.0 : 1.15);
}

grim_status_t launch_direct(const grim_bcr* h, const SpmmArgs& a, cudaStream_t s) {
  if (!direct_path_supported(h, a)) return GRIM_ERR_UNSUPPORTED;
  DParams p;
  p.w.head = h->d_rc_head; p.w.blob = h->d_rc_blob; p.w.nbc = (int)h->nbc; p.w.bw = h->bw;
  p.band_order = h->d_band_order; p.nbr = (int)h->nbr; p.M = (int)h->M; p.bh = h->bh;
  p.a = a;
  const int BHc = h->bh <= 4 ? 4 : (h->bh <= 8 ? 8 : 16);
  int nc, parts;
  if (a.tile_n > 32 && direct_choice(a.tile_n)) {
    nc = a.tile_n % 32; parts = a.tile_n / 256;
  } else {
    const Shape shape = shape_for(h, a);
    nc = shape.nc; parts = shape.parts;
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
