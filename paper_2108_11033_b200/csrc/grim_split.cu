// fp32 products and convolutions on the tensor cores (tcgen05), every operand split into three bf16 numbers: large right-hand
// sides of fp32 handles (Section 3.1: every layer is a GEMM; Sections 4.3 - 4.5: compact weights expanded only on chip,
// the expanded input of a convolution never produced in memory).
//
// A value v is written as b1 + b2 + b3, b1 = bf16(v), b2 = bf16(v - b1), b3 = v - b1 - b2: three times eight bits, so that the sum is v
// itself, all 24 bits of it, whatever its neighbours are (bf16 has fp32's exponents; nothing is scaled).  A product is the sum of the six
// products of parts that are not below its own last bit (b1 b1, b1 b2, b2 b1, b2 b2, b1 b3, b3 b1; what is left out is below 2^-25 of it),
// the small ones first, which the tensor core sums in fp32.  Its additions truncate, so a sum only runs over 64 values of k (16 at a
// time) there; the sums of those chunks are added up in registers, rounded to nearest.  (Measured: products and sums down to 2^-149 are
// kept as fp32 multiplies keep them.)  Columns of X with infinities, NaN or numbers so small or large that parts or sums of products leave
// the range (kSplitLeast and the following) are worked out again with fp32 multiplies (row_walk), product by kept product; handles with such
// weights have no layout for this kernel.
// (Two fp16 numbers and a scale per column and 64 values of k need half the multiplies, but lose what is much smaller than its
// neighbours in k: a row of a pruned matrix that does not keep the large ones then consists of what was lost.)
//
// The multiply is transposed: 128 columns of X are the rows of the tensor core's tile, 128 rows of W its columns.  A thread
// that owns a column of X then splits it and adds it up without looking at its
// neighbours; loads and stores of 32 neighbouring columns are whole lines; and the activations go from registers to tensor memory
// (the A operand is read from there), so that shared memory, whose bandwidth bounds the bf16 kernels, holds weights only.
//
// Per thread block: one thread requests packed weights (bulk copies), another 64 x 128 values of X (TMA, two K tiles ahead), four
// warps expand the weights (a list of them and their places, made when the matrix is packed) into three swizzled tiles
// of a 64-wide K tile, two groups of four warps split activations, K tiles in turn, one thread issues the multiplies (24
// per K tile), eight warps add up.  With few tiles the blocks of a cluster share one, each multiplying a part of K; the sums
// meet over distributed shared memory.
//
// What bounds it: some 2200 cycles a K tile, 1536 of them the multiplies' at their nominal rate (two stages, so that a K tile's operands
// are written while the tile before it is multiplied): 8192^2, rate 8, N = 1024, 128 K tiles in three rounds and a half, 524 us, where six
// dense bf16 products at the rate that a library's product reaches take 503.  In loops of seconds the card is at its power limit: 593,
// and 597 at that product's sustained rate.  (The slab kernel, bound by its fp32 multiplies: 665.)  Convolutions read pixels one by one and
// take 1.55 us a K tile, matrices 1.15.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "grim_device.cuh"
#include "grim_internal.h"
#include "grim_rowwalk.cuh"

namespace grim {
namespace {

using namespace ptx;

constexpr int kTile = 128;                        // rows of W and columns of X per thread block
constexpr int kK = 64;                            // K per stage, and per sum in tensor memory
constexpr int kStages = 2;                        // a converting group's own each
constexpr int kParts = 3;                         // bf16 numbers to a value
constexpr int kXBytes = kK * kTile * 4;            // a K tile of activations as TMA brings it
constexpr int kPartBytes = kTile * kK * 2;        // one expanded tile of 16-bit weights
constexpr int kStageBytes = kParts * kPartBytes;
constexpr int kPartCols = kK / 2, kStageCols = kParts * kPartCols;  // columns of tensor memory that a part, a stage of activations takes
constexpr int kMaxRec = 8;                        // ring of packed weights
constexpr int kExpand0 = 4, kConvert0 = 8, kSum0 = 16, kWarps = 24;  // first warps of the roles; 0: copies, 1: tensor core
constexpr int kThreads = 32 * kWarps;
// Registers per thread of the roles.  The block is launched with 80 x 768; what the first two give back the others take.
constexpr int kRegsMisc = 40, kRegsExpand = 56, kRegsConvert = 104, kRegsSum = 88;
static_assert(kRegsMisc + kRegsExpand + 2 * kRegsConvert + 2 * kRegsSum <= 6 * 80, "more registers than the block is launched with");
constexpr int kMaxParts = 8;                      // thread blocks that share a tile
// shared memory: barriers and tables, stages, packed weights.  After the multiplies the stages hold the exchange of the
// sums ([part][row][column]), behind it columns that were worked out again, behind those the walk's weight buffers.
constexpr int kBars = 0, kTmem = 512, kAbort = 516, kAnyFlag = 520, kMeta = 1024;           // kMeta: [record] entries
constexpr int kFlagTiles = 256;                   // K tiles of a block whose flagged columns are told apart
constexpr int kRow = kMeta + kMaxRec * 4, kFlags = kRow + kTile * 4, kTaps = kFlags + kFlagTiles * kTile / 8;  // [128] rows; [K tile][128] flags; [2][2][64] kernel positions
constexpr int kHdr = (kTaps + 2 * 2 * kK * 8 + 1023) / 1024 * 1024;
constexpr int kExchangeBytes = (kTile + kMaxParts) * kTile * 4, kPatchBytes = kTile * kTile * 4;
constexpr int kTailBytes = kExchangeBytes + kPatchBytes + 8 * kWalkBufFloats * 4;

struct SplitParams {
  RowWalk w;
  const RcStage* stage;
  const uint8_t* blob;
  const uint32_t* band_order;
  unsigned* status;
  int nbr, M, K, nbc, nkt;
  int mtiles, parts, kt_per;
  int nrec, tma;
  uint32_t rec_stride;
  unsigned spin_limit;
  int tile0;  // first tile of this launch
  SpmmArgs a;
};

// K-major tile with rows of 128 bytes in the 128-byte swizzle, groups of eight rows 1 KiB apart.
__device__ __forceinline__ uint64_t tile_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// fp32 sums, bf16 x bf16, both operands K-major, 128 x 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t bdesc, uint32_t accumulate) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}"
               ::"r"(d), "r"(a_tmem), "l"(bdesc), "r"(kIdesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The next part of two values: their bf16 numbers, which leave them.  PAIR: both subtractions in one instruction, which wants
// neighbouring registers (the convolution's loop has none to spare for that).
template <bool PAIR>
__device__ __forceinline__ uint32_t take_part(unsigned long long& x) {
  const float x0 = __uint_as_float((uint32_t)x), x1 = __uint_as_float((uint32_t)(x >> 32));
  const __nv_bfloat162 b = __floats2bfloat162_rn(x0, x1);
  const uint32_t u = *reinterpret_cast<const uint32_t*>(&b);
  const float b0 = __uint_as_float(u << 16), b1 = __uint_as_float(u & 0xFFFF0000u);
  if (PAIR) walk_ffma2(x, walk_pair(b0, b1), walk_pair(-1.f, -1.f));
  else x = walk_pair(x0 - b0, x1 - b1);
  return u;
}

// Entries v of a record (grim_internal.h), eight of them: their parts and places.
struct Entries {
  uint32_t part[kParts][4], off[4];
  __device__ __forceinline__ void load(uint32_t rec, uint32_t n, uint32_t v) {
    const uint4 a = lds128(rec + v * 32u), b = lds128(rec + v * 32u + 16u), at = lds128(rec + n * 4u + v * 16u);
    unsigned long long w[4] = {(unsigned long long)a.y << 32 | a.x, (unsigned long long)a.w << 32 | a.z,
                               (unsigned long long)b.y << 32 | b.x, (unsigned long long)b.w << 32 | b.z};
    off[0] = at.x; off[1] = at.y; off[2] = at.z; off[3] = at.w;
#pragma unroll
    for (int l = 0; l < kParts; ++l)
#pragma unroll
      for (int i = 0; i < 4; ++i) part[l][i] = take_part<true>(w[i]);
  }
  __device__ __forceinline__ void store(uint32_t tile) const {  // into the three tiles there
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t to0 = tile + (off[i] & 0xFFFFu), to1 = tile + (off[i] >> 16);
#pragma unroll
      for (int l = 0; l < kParts; ++l) {
        sts16(to0 + l * kPartBytes, part[l][i]);
        sts16(to1 + l * kPartBytes, part[l][i] >> 16);
      }
    }
  }
};

// Writes the record of a tile: a thread block per tile, a warp per block of the matrix, a lane per kept weight.
constexpr int kBuildThreads = 128;
__global__ void __launch_bounds__(kBuildThreads) build_records_kernel(RowWalk w, const RcStage* __restrict__ stage,
                                                                      int nbr, int bh, uint8_t* __restrict__ out) {
  __shared__ uint32_t first[kTile / 4 * (kK / 16)];   // entries before each block
  __shared__ uint32_t size[32];                       // entries that fall into each bank
  __shared__ uint16_t rank_of[kTile * kK];            // ... and how many of its bank came before an entry
  const int kt = blockIdx.x, mt = blockIdx.y, nkt = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const RcStage se = stage[(int64_t)mt * nkt + kt];
  if (se.bytes == 0) return;
  const int NB = kTile / bh, J = kK / w.bw, blocks = NB * J;
  auto head_of = [&](int i) {
    const int pos = mt * NB + i / J, j = kt * J + i % J;
    RcHead h{0u, 0u, {0u, 0u}};
    if (pos < nbr && j < w.nbc) h = w.head[(int64_t)pos * w.nbc + j];
    return h;
  };
  if (tid < 32) size[tid] = 0;
  for (int i = tid; i < blocks; i += kBuildThreads) {
    const RcHead h = head_of(i);
    first[i] = (uint32_t)(__popc(rc_head_rows(h.rows_kc)) * rc_head_kc(h.rows_kc));
  }
  __syncthreads();
  if (tid == 0) {
    uint32_t sum = 0;
    for (int i = 0; i < blocks; ++i) { const uint32_t n = first[i]; first[i] = sum; sum += n; }
  }
  __syncthreads();
  const uint32_t n = se.bytes / 6;  // a multiple of eight: the first entry is repeated
  uint32_t total = 0;
  // position of an entry that is number r of its bank's: number r of all banks come before, then those of the banks to the left
  auto position = [&](uint32_t bank, uint32_t r) {
    uint32_t p = 0;
    for (uint32_t b = 0; b < 32; ++b) p += min(size[b], r) + (b < bank && size[b] > r ? 1u : 0u);
    return p;
  };
  // entry number p of a run of 256 is stored by lane p % lanes as its (p / lanes)-th of eight
  auto put = [&](uint32_t p, uint32_t val, uint32_t off) {
    const uint32_t run = p & ~255u, i = p - run, lanes = min(256u, n - run) >> 3, at = run + 8u * (i % lanes) + i / lanes;
    reinterpret_cast<uint32_t*>(out + (size_t)se.off16 * 16)[at] = val;
    reinterpret_cast<uint16_t*>(out + (size_t)se.off16 * 16 + (size_t)n * 4)[at] = (uint16_t)off;
  };
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1)
      for (int b = 0; b < 32; ++b) total += size[b];
    for (int i = warp; i < blocks; i += kBuildThreads / 32) {
      const RcHead h = head_of(i);
      const uint32_t rows = rc_head_rows(h.rows_kc);
      const int kc = rc_head_kc(h.rows_kc), kr = __popc(rows), nch = (kc + kRcChunk - 1) / kRcChunk;
      const uint8_t* rec = w.blob + (size_t)h.rec16 * 16;
      const float* wv = reinterpret_cast<const float*>(rec + ((8 + nch * kRcChunk + 15) & ~15));
      for (int e = lane; e < kr * kc; e += 32) {
        const int a = e / kc, c = e - a * kc;
        uint32_t m = rows;
        for (int k = 0; k < a; ++k) m &= m - 1;
        const int r = __ffs(m) - 1, row = (i / J) * bh + r, col = (i % J) * w.bw + rec[8 + c];
        const uint32_t off = (uint32_t)row * 128u + (((uint32_t)(col >> 3) ^ (uint32_t)(row & 7)) << 4) + (uint32_t)(col & 7) * 2u;
        const uint32_t bank = (off >> 2) & 31u, id = first[i] + (uint32_t)e;
        if (pass == 0) {
          rank_of[id] = (uint16_t)atomicAdd(&size[bank], 1u);
        } else {
          const uint32_t val = __float_as_uint(wv[((c / kRcChunk) * kr + a) * kRcChunk + c % kRcChunk]);
          put(position(bank, rank_of[id]), val, off);
          if (id == 0)
            for (uint32_t p = total; p < n; ++p) put(p, val, off);
        }
      }
    }
    __syncthreads();
  }
}

// What the split cannot hold, product by kept product: flagged columns of a K tile (bits of flags[K tile][column]), where the parts have
// been left out, rows of the tile's bands worker, worker + 8, ..., are added to patch[row][column].  A block of more than
// kFlagTiles K tiles has one set of flags, and its flagged columns are worked out again over all of its K.  (One row of X of 8192 x 1024
// that is not finite: 8192^2, 8 x 32: 0.74 ms beside 0.54; worked out over the whole of K: 5.7 ms.)
template <int BH, int CONV>
__device__ __forceinline__ void exact_columns(const SplitParams& p, int tile, int64_t q0, int kt0, int n, int worker, int lane, const uint32_t* flags,
                                           float* patch, float* wbuf) {
  const bool apart = n <= kFlagTiles;
  const int J = kK / p.w.bw;
  for (int i = 0; i < (apart ? n : 1) * (kTile / 32); ++i) {
    const int it = i / (kTile / 32), c0 = i % (kTile / 32) * 32;
    const uint32_t flagged = flags[i];
    if (!flagged) continue;
    const bool mine = (flagged >> lane) & 1u;
    RowRange w;
    w.head = p.w.head; w.blob = p.w.blob; w.bw = p.w.bw;
    w.j0 = (kt0 + it) * J; w.stride = p.nbc; w.nbc = min((apart ? 1 : n) * J, p.nbc - w.j0);
    WalkCols<1, 1> wc;
    walk_setup<1, 1, float, CONV>(p.a, q0 + c0, lane, wc);
    for (int lb = worker; lb < kTile / BH; lb += 8) {
      const int pos = tile * (kTile / BH) + lb;
      if (pos >= p.nbr) break;
      float acc[BH];
      unsigned long long unused[1][1];
#pragma unroll
      for (int r = 0; r < BH; ++r) acc[r] = 0.f;
      row_walk<BH, 1, 1, float, CONV, true>(w, p.a, pos, 0, 1, wc, wbuf, lane, acc, unused, [] {});
#pragma unroll
      for (int r = 0; r < BH; ++r) {
        float* at = patch + (lb * BH + r) * kTile + c0 + lane;
        if (mine) *at = apart ? *at + acc[r] : acc[r];
      }
      __syncwarp();
    }
  }
}

template <int N>
__device__ __forceinline__ void more_registers() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void fewer_registers() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

template <int BH, int CONV>
__global__ void __launch_bounds__(kThreads, 1) bcr_split_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ SplitParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  // (the offset of the 1 KiB boundary is the same in all blocks of a cluster)
  uint8_t* smem = align_smem(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kBars);  // both operands of a K tile are in place
  uint64_t* empty = full + kStages;                            // its multiplies are done
  uint64_t* sum_full = empty + kStages;                        // [2] a chunk's sums are complete
  uint64_t* sum_empty = sum_full + 2;                          // [2] ... and have been read
  uint64_t* rec_full = sum_empty + 2;
  uint64_t* rec_empty = rec_full + kMaxRec;
  uint64_t* x_full = rec_empty + kMaxRec;                      // [2] activations have landed
  uint64_t* x_empty = x_full + 2;                              // [2] ... and are in registers
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + kAbort);
  int* s_any = reinterpret_cast<int*>(smem + kAnyFlag);
  uint32_t* s_meta = reinterpret_cast<uint32_t*>(smem + kMeta);
  int* s_row = reinterpret_cast<int*>(smem + kRow);
  uint32_t* s_flags = reinterpret_cast<uint32_t*>(smem + kFlags);
  uint8_t* stages = smem + kHdr;
  uint8_t* xs = stages + kStages * kStageBytes;
  uint8_t* recs = xs + (p.tma ? 2 * kXBytes : 0);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const SpmmArgs& a = p.a;
  const int parts = p.parts, part = parts > 1 ? (int)cluster_ctarank() : 0;
  const int t = p.tile0 + (int)blockIdx.x / parts, mt = t % p.mtiles;
  const int64_t q0 = (int64_t)(t / p.mtiles) * kTile;
  const int kt0 = part * p.kt_per, n = min(p.kt_per, p.nkt - kt0);  // this block's K tiles
  constexpr int NB = kTile / BH;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full + s, 8); mbar_init(empty + s, 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(sum_full + s, 1); mbar_init(sum_empty + s, 8); mbar_init(x_full + s, 1); mbar_init(x_empty + s, 4); }
    for (int s = 0; s < kMaxRec; ++s) { mbar_init(rec_full + s, 1); mbar_init(rec_empty + s, 4); }
    *s_abort = 0;
    *s_any = 0;
    fence_mbar_init();
  }
  if (tid < kTile) {
    const int pos = mt * NB + tid / BH;
    int row = -1;
    if (pos < p.nbr) row = (int)p.band_order[pos] * BH + (tid & (BH - 1));
    if (row >= p.M) row = -1;
    s_row[tid] = row;
  }
  for (int i = tid; i < kFlagTiles * kTile / 32; i += kThreads) s_flags[i] = 0u;
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(smem + kTmem)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + kTmem);
  const uint32_t tmem_a = tmem + 256;  // columns 0 .. 255: two chunks' sums; then 96 per stage

  // Every role goes through the same block barriers at its own end (registers are dealt by role, so the ends are not shared).
  // After the first all multiplies are done and the stages are free.
  auto end_of_loop = [&](bool failed, int fail_site) {
    if (__any_sync(0xffffffffu, failed)) {
      *s_abort = 1;
      if (fail_site) atomicOr(p.status, (unsigned)GRIM_ERR_TIMEOUT | (1u << (8 + fail_site)));
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*s_abort) let_copies_land();
  };
  auto rest = [&]() {  // of the barriers, for the roles that have nothing to do between them
    if (*s_any && !*s_abort) { __syncthreads(); __syncthreads(); }
    if (parts > 1) { cluster_sync_all(); cluster_sync_all(); }
    __syncthreads();
  };
  float* exchange = reinterpret_cast<float*>(stages);
  float* patch = reinterpret_cast<float*>(stages + kExchangeBytes);
  bool failed = false;
  int fail_site = 0;
  if (warp < kExpand0) {
    fewer_registers<kRegsMisc>();
    if (warp == 0 && elect_one()) {
      // ---------------------------------------------------------------- packed weights
      const RcStage* stage = p.stage + (int64_t)mt * p.nkt + kt0;
      RcStage next = stage[0];
      int rs = 0;
      unsigned par = 1;
      for (int it = 0; it < n; ++it) {
        const RcStage se = next;
        if (it + 1 < n) next = stage[it + 1];
        if (!mbar_wait(rec_empty + rs, par, p.spin_limit, s_abort, 20)) { failed = true, fail_site = 1; break; }
        s_meta[rs] = se.bytes / 6;
        mbar_arrive_expect_tx(rec_full + rs, se.bytes);
        if (se.bytes) bulk_load(recs + (size_t)rs * p.rec_stride, p.blob + (size_t)se.off16 * 16, se.bytes, rec_full + rs);
        if (++rs == p.nrec) { rs = 0; par ^= 1u; }
      }
    } else if (warp == 1 && elect_one()) {
      // ---------------------------------------------------------------- tensor core
      int s = 0;
      unsigned par = 0;
      for (int it = 0; it < n; ++it) {
        const int buf = it & 1;
        if (!mbar_wait_tight(full + s, par, p.spin_limit << 2, s_abort)) { failed = true, fail_site = 2; break; }
        if (!mbar_wait_tight(sum_empty + buf, (unsigned)((it >> 1) + 1) & 1u, p.spin_limit << 2, s_abort)) { failed = true, fail_site = 3; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem + (uint32_t)buf * kTile, xa = tmem_a + (uint32_t)s * kStageCols;
        const uint64_t w = tile_desc(smem_u32(stages + s * kStageBytes));
        // the small products first; 16 values of k: eight columns of tensor memory, 32 bytes of a tile's rows
        auto products = [&](int of_x, int of_w, bool first) {
#pragma unroll
          for (int k = 0; k < 4; ++k) mma_ts(d, xa + of_x * kPartCols + 8u * k, w + of_w * (kPartBytes >> 4) + 2u * k, !(first && k == 0));
        };
        products(2, 0, true);
        products(0, 2, false);
        products(1, 1, false);
        products(1, 0, false);
        products(0, 1, false);
        products(0, 0, false);
        commit(empty + s);
        commit(sum_full + buf);
        if (++s == kStages) { s = 0; par ^= 1u; }
      }
    } else if (warp == 3 && p.tma && elect_one()) {
      // ---------------------------------------------------------------- activations, two K tiles ahead
      asm volatile("griddepcontrol.wait;" ::: "memory");
      for (int it = 0; it < n; ++it) {
        const int g = it & 1;
        if (!mbar_wait(x_empty + g, (unsigned)((it >> 1) + 1) & 1u, p.spin_limit, s_abort, 20)) { failed = true, fail_site = 8; break; }
        mbar_arrive_expect_tx(x_full + g, kXBytes);
        tma_load_2d(xs + g * kXBytes, &tm_x, (int)q0, (kt0 + it) * kK, x_full + g);
      }
    }
    __syncwarp();
    end_of_loop(failed, fail_site);
    rest();
    if (warp == 2) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
  } else if (warp < kConvert0) {
    // ------------------------------------------------------------------ weights
    fewer_registers<kRegsExpand>();
    const int gw = warp & 3;
    int rs = 0;
    unsigned rpar = 0, par = 1;  // (a fresh barrier counts as emptied one round before)
    int s = 0;
    for (int it = 0; it < n; ++it, s = s + 1 == kStages ? 0 : s + 1, par ^= s == 0 ? 1u : 0u) {
      // (a thread's first entries, mostly all that it has, are split before the stage is free)
      if (!failed && !__all_sync(0xffffffffu, mbar_wait(rec_full + rs, rpar, p.spin_limit, s_abort, 32))) failed = true, fail_site = 5, *s_abort = 1;
      const uint32_t rec = smem_u32(recs + (size_t)rs * p.rec_stride), tile = smem_u32(stages + s * kStageBytes), wt = (uint32_t)(gw * 32 + lane);
      const uint32_t n = failed ? 0u : s_meta[rs];
      Entries e;
      if (wt < (n >> 3)) e.load(rec, n, wt);
      if (!failed && !__all_sync(0xffffffffu, mbar_wait(empty + s, par, p.spin_limit, s_abort, 0))) failed = true, fail_site = 4, *s_abort = 1;
      if (!failed) {
#pragma unroll
        for (int i = 0; i < kStageBytes / 16 / 128; ++i) sts128(tile + (wt + i * 128) * 16u, 0u, 0u, 0u, 0u);
      }
      named_barrier(1, 128);  // (also for a warp that has given up: the others may be waiting here)
      if (failed) continue;
      if (wt < (n >> 3)) e.store(tile);
      for (uint32_t v = wt + 128u; v < (n >> 3); v += 128u) {
        e.load(rec, n, v);
        e.store(tile);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(full + s);
        mbar_arrive(rec_empty + rs);
      }
      if (++rs == p.nrec) { rs = 0; rpar ^= 1u; }
    }
    end_of_loop(failed, fail_site);
    rest();
  } else if (warp < kSum0) {
    // ------------------------------------------------------------------ activations
    more_registers<kRegsConvert>();
    const int grp = (warp - kConvert0) >> 2, quarter = warp & 3, col = quarter * 32 + lane;
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    WalkCols<1, 1> wc;
    walk_setup<1, 1, float, CONV>(a, q0 + quarter * 32, lane, wc);
    const bool valid = q0 + col < a.ncols;
    const float* X = static_cast<const float*>(wc.ptr[0]);
    int2* taps = reinterpret_cast<int2*>(smem + kTaps) + grp * 2 * kK;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // what earlier launches in the stream wrote is complete
    const int s = grp;  // (two groups, two stages)
    unsigned par = 1;
    for (int it = grp; it < n; it += 2, par ^= 1u) {
      const int k0 = (kt0 + it) * kK;
      union { float x[kK]; unsigned long long x2[kK / 2]; };
      if (!CONV && p.tma) {
        if (!failed && !__all_sync(0xffffffffu, mbar_wait(x_full + grp, (unsigned)(it >> 1) & 1u, p.spin_limit, s_abort, 32))) failed = true, fail_site = 9, *s_abort = 1;
        const float* src = reinterpret_cast<const float*>(xs + grp * kXBytes) + col;  // (zeros past the last row and column)
#pragma unroll
        for (int k = 0; k < kK; ++k) x[k] = src[k * kTile];
      } else if (CONV) {
        // k -> offset in the input and kernel position (none that is inside, past the last k)
        int2* tp = taps + ((it >> 1) & 1) * kK;
        const int i = quarter * 32 + lane;
        if (i < kK) {
          const int k = k0 + i, khw = a.KH * a.KW, c = k / khw, rest = k - c * khw, kh = rest / a.KW, kw = rest - kh * a.KW;
          tp[i] = k < p.K ? make_int2((c * a.H + kh) * a.W + kw, (int)((1u << kh) | (1u << (16 + kw)))) : make_int2(0, -1);
        }
        if (grp) named_barrier(3, 128); else named_barrier(2, 128);
#pragma unroll
        for (int k = 0; k < kK; ++k) {
          const int2 tk = tp[k];
          x[k] = 0.f;
          if ((wc.valid[0] & (unsigned)tk.y) == (unsigned)tk.y) x[k] = __ldg(X + tk.x);
        }
      } else {
        const float* xk = X + (int64_t)k0 * a.x_sk;
        if (k0 + kK <= p.K) {
#pragma unroll
          for (int k = 0; k < kK; ++k, xk += a.x_sk) x[k] = __ldg(xk);
        } else {
#pragma unroll
          for (int k = 0; k < kK; ++k, xk += a.x_sk) x[k] = k0 + k < p.K ? __ldg(xk) : 0.f;
        }
      }
      if (!failed && !__all_sync(0xffffffffu, mbar_wait(empty + s, par, p.spin_limit, s_abort, 0))) failed = true, fail_site = 6, *s_abort = 1;
      if (failed) continue;  // (as above)
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");  // (another thread's multiplies have read what is overwritten below)
      // the largest and the smallest magnitude but zero among the first parts, in pairs of 16 bits: less one and with the sign bit
      // set a zero becomes the smallest number without a sign and the largest with one
      uint32_t largest = 0u, least = 0x7FFF7FFFu;
      const uint32_t to = tmem_a + lanes + (uint32_t)s * kStageCols;
#pragma unroll
      for (int l = 0; l < kParts; ++l)
#pragma unroll
        for (int h = 0; h < kPartCols; h += 16) {
          uint32_t part[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            part[i] = take_part<!CONV>(x2[h + i]);
            if (l == 0) {
              const uint32_t b = (part[i] | 0x80008000u) - 0x00010001u;
              largest = __vmaxu2(largest, b);
              least = __vmins2(least, b);
            }
          }
          tmem_st16(to + l * kPartCols + h, part);
          if (!CONV && p.tma && l == 0 && h) {  // (all of x is in registers)
            __syncwarp();
            if (lane == 0) mbar_arrive(x_empty + grp);
          }
        }
      const int low = min((int)(int16_t)(least & 0xFFFFu), (int)(int16_t)(least >> 16));
      const bool bad = max(largest & 0xFFFFu, largest >> 16) >= 0x7FFFu + (kSplitBeyondX >> 16) || low < -0x8001 + (int)(kSplitLeast >> 16);
      const uint32_t flagged = __ballot_sync(0xffffffffu, bad && valid);
      if (flagged) {  // their parts are left out
        if (lane == 0) {
          atomicOr(s_flags + (n <= kFlagTiles ? it : 0) * (kTile / 32) + quarter, flagged);
          *s_any = 1;
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
#pragma unroll 1
        for (int c = 0; c < kStageCols; c += 16) {
          uint32_t part[16];
          tmem_ld16(to + c, part);
#pragma unroll
          for (int i = 0; i < 16; ++i) part[i] = bad ? 0u : part[i];
          tmem_st16(to + c, part);
        }
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(full + s);
    }
    end_of_loop(failed, fail_site);
    if (*s_any && !*s_abort) {
      __syncthreads();  // the sums lie in `patch`
      float* wbuf = reinterpret_cast<float*>(stages + kExchangeBytes + kPatchBytes) + (warp - kConvert0) * kWalkBufFloats;
      exact_columns<BH, CONV>(p, mt, q0, kt0, n, warp - kConvert0, lane, s_flags, patch, wbuf);
      __syncthreads();
    }
    if (parts > 1) { cluster_sync_all(); cluster_sync_all(); }
    __syncthreads();
  } else {
    // ------------------------------------------------------------------ sums of the chunks
    more_registers<kRegsSum>();
    const int quarter = warp & 3, half = (warp - kSum0) >> 2, col = quarter * 32 + lane;
    const uint32_t from = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 64);
    unsigned long long acc[32];  // a column of X, 64 rows of the tile, in pairs
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0ull;
    for (int it = 0; it < n; ++it) {
      const int buf = it & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(sum_full + buf, (unsigned)(it >> 1) & 1u, p.spin_limit << 2, s_abort, 32))) { failed = true, fail_site = 7; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t v[16];
        tmem_ld16(from + (uint32_t)(buf * kTile + c * 16), v);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[8 * c + i]) : "l"(walk_pair(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]))));
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(sum_empty + buf);
    }
    end_of_loop(failed, fail_site);
    const int64_t q = q0 + col;
    // (through shared memory, so that what follows is loops and no more registers)
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      patch[(half * 64 + 2 * i) * kTile + col] = __uint_as_float((unsigned)acc[i]);
      patch[(half * 64 + 2 * i + 1) * kTile + col] = __uint_as_float((unsigned)(acc[i] >> 32));
    }
    if (*s_any && !*s_abort) {
      __syncthreads();  // flagged columns are worked out again by the warps that read the activations
      __syncthreads();
    }
    const bool writes = q < a.ncols && !*s_abort;
    auto value = [&](int r) { return patch[r * kTile + col]; };
    int64_t at_q = q * a.y_sq, row_stride = a.y_sr;
    if (CONV) {
      row_stride = (int64_t)a.OH * a.OW;
      const int64_t img = q / row_stride;
      at_q = img * p.M * row_stride + (q - img * row_stride);
    }
    float* out = static_cast<float*>(a.Y) + at_q;
    auto store = [&](int row, float v) {  // (row is the same in all lanes)
      if (a.relu) v = fmaxf(v, 0.f);
      if (writes) out[(int64_t)row * row_stride] = v;
    };
    if (parts == 1) {
#pragma unroll 4
      for (int r = half * 64; r < half * 64 + 64; ++r) {
        const int row = s_row[r];
        if (row >= 0) store(row, value(r) + (a.bias ? __ldg(a.bias + row) : 0.f));
      }
    } else {
      // Every block of the cluster owns some of the tile's rows: each sends its sums of them to their owner, who adds them up.
      const int nr = (kTile + parts - 1) / parts;
      cluster_sync_all();
      const uint32_t mine = smem_u32(exchange) + ((uint32_t)part * (uint32_t)nr * kTile + (uint32_t)col) * 4u;
      for (int r = half * 64; r < half * 64 + 64;) {
        const int owner = r / nr, first = owner * nr, end = min(first + nr, half * 64 + 64);
        uint32_t to;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(mine + (uint32_t)(r - first) * (kTile * 4)), "r"(owner));
#pragma unroll 4
        for (; r < end; ++r, to += kTile * 4) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to), "f"(value(r)) : "memory");
      }
      __syncwarp();
      cluster_sync_all();
#pragma unroll 2
      for (int r = half; r < min(nr, kTile - part * nr); r += 2) {
        const int row = s_row[part * nr + r];
        if (row < 0) continue;
        // what the additions round off is summed on the side: otherwise a third of the whole error
        float sum = 0.f, off = 0.f;
        auto add = [&](float v) {
          const float t = sum + v, w = t - sum;
          off += (sum - (t - w)) + (v - w);
          sum = t;
        };
        for (int s = 0; s < parts; ++s) add(exchange[(s * nr + r) * kTile + col]);
        if (a.bias) add(__ldg(a.bias + row));
        store(row, isfinite(off) ? sum + off : sum);
      }
    }
    __syncthreads();
  }
}

uint32_t rec_stride_of(const grim_bcr* h) { return (h->sp_max_rec + 127u) & ~127u; }
size_t smem_need(const grim_bcr* h, int nrec, bool tma) {
  return 1024 + kHdr + std::max<size_t>((size_t)kStages * kStageBytes + (tma ? 2 * kXBytes : 0) + (size_t)nrec * rec_stride_of(h), kTailBytes);
}
int rec_slots(const grim_bcr* h, bool tma) {
  for (int n = kMaxRec; n >= 2; --n)
    if (smem_need(h, n, tma) <= 227 * 1024) return n;
  return 0;
}

template <int BH>
cudaError_t launch_rows(const CUtensorMap& tm, const SplitParams& p, unsigned grid, size_t smem, cudaStream_t s) {
  auto kern = p.a.conv ? bcr_split_kernel<BH, 1> : bcr_split_kernel<BH, 0>;
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)p.parts;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.parts > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, tm, p);
}

}  // namespace

// Fills h->d_sp_blob, whose records h->d_sp_stage names, from the row-chunk layout.
grim_status_t build_split_records(grim_bcr* h) {
  RowWalk w;
  w.head = h->d_rc_head; w.blob = h->d_rc_blob; w.nbc = (int)h->nbc; w.bw = h->bw;
  build_records_kernel<<<dim3((unsigned)h->sp_ktiles, (unsigned)h->sp_mtiles), kBuildThreads>>>(w, h->d_sp_stage, (int)h->nbr, h->bh, h->d_sp_blob);
  return cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(nullptr) == cudaSuccess ? GRIM_OK : GRIM_ERR_CUDA;
}

bool split_path_supported(const grim_bcr* h, const SpmmArgs& a) {
  if (h->device < 0 || h->dtype != GRIM_F32 || !h->d_sp_blob || !h->d_rc_head || !h->d_status || !rec_slots(h, false)) return false;
  if (a.x_dtype != GRIM_F32 || a.y_dtype != GRIM_F32 || a.ncols <= 0) return false;
  const int64_t tiles = (h->M + kTile) / kTile * ((a.ncols + kTile - 1) / kTile);
  if (a.ncols > (int64_t(1) << 31) - 512 || tiles > (int64_t(1) << 27)) return false;
  if (!a.conv && a.x_sk * 4 >= (int64_t(1) << 32)) return false;
  if (a.conv && (a.KH > 16 || a.KW > 16 || (int64_t)a.C * a.H * a.W >= (int64_t(1) << 31))) return false;
  return true;
}

namespace {
// Whole rounds of tiles, a thread block each, and the tiles of the last round, which would leave SMs idle: as many blocks of a
// cluster to each as run at once with K tiles for all of them (clusters of n that run at once on 148 SMs).  8192^2, N = 1024: 512
// tiles are three rounds and 68 pairs, 5 % less than four rounds.
struct Plan { int64_t whole, tail; int parts, kt_per; };
Plan plan_for(const grim_bcr* h, const SpmmArgs& a) {
  static const int at_once[kMaxParts + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
  const int64_t tiles = h->sp_mtiles * ((a.ncols + kTile - 1) / kTile);
  const int nkt = (int)h->sp_ktiles, sms = sm_count(h->device);
  Plan pl{tiles - tiles % sms, tiles % sms, 1, nkt};
  for (int n = 2; n <= kMaxParts; ++n) {
    const int per = (nkt + n - 1) / n;
    if (pl.tail * 148 <= (int64_t)at_once[n] * sms && per >= 2 && per < pl.kt_per && (n - 1) * per < nkt) pl.parts = n, pl.kt_per = per;
  }
  if (pl.whole && nkt - pl.kt_per < 6) pl = {tiles, 0, 1, nkt};  // (a second launch costs a few us)
  return pl;
}
// rows that TMA can fetch come through shared memory, others (and a convolution's pixels) are read by the threads that split them
bool rows_by_tma(const grim_bcr* h, const SpmmArgs& a) {
  return !a.conv && a.x_sq == 1 && a.x_sk % 4 == 0 && reinterpret_cast<uintptr_t>(a.X) % 16 == 0 && rec_slots(h, true) >= 3;
}
}  // namespace

// Estimate in us, fitted to 119 products and 81 convolutions of 17 .. 8192 rows and 64 .. 12,800 columns of W and N of 17 .. 105,000, rates
// 4 to 16: nine in ten within 15 %.
double split_time(const grim_bcr* h, const SpmmArgs& a) {
  const Plan pl = plan_for(h, a);
  const int sms = sm_count(h->device);
  const double kt = a.conv ? 1.55 : (rows_by_tma(h, a) ? 1.15 : 1.2), ends = a.conv ? 8.0 : 6.0;
  double t = (a.conv ? 3.0 : 5.0) + (double)((pl.whole + sms - 1) / sms) * ((double)h->sp_ktiles * kt + ends);
  if (pl.tail) t += pl.kt_per * kt + ends + (pl.parts > 1 ? (a.conv ? 2.0 : 1.0) : 0.0) + (pl.whole && pl.parts > 1 ? 3.0 : 0.0);
  return t;
}

// Errors, squared, as fractions of the result's norm, fitted (with 10 % on this kernel's side) to fp64 comparisons of the products and
// convolutions above: weights and activations of both signs, and all of one sign, where roundings of fp32 sums average out over
// the threads that share a row's sum and the tensor core's truncations do not.  Here: truncations and the sums of chunks.  fp32 kernels: the
// square root of the products that one thread adds up (convolutions, half of whose inputs ReLU has made zero: of fewer), and
// the sum of the threads' sums.  Where this says yes the error is 0.24 to 0.97 times that of the kernel whose place is taken, 0.6 on average
// (8192^2, N = 1024: 1.9e-7 against 5.1e-7; 512 -> 512 channels, 28 x 28, one image: 0.85e-7 against 1.26e-7), with one sign 0.25 to 1.11 times (1.4e-7
// against 3.8e-7; 0.58e-7 against 0.67e-7), or below the rounding of a single result, 2^-24.
// Up to 16 columns other kernels run, which spread a row over 32 lanes: no comparison, no yes.
bool split_precise(const grim_bcr* h, const SpmmArgs& a) {
  if (a.ncols <= kSkinnyMaxN || !split_path_supported(h, a)) return false;
  const double direct = direct_path_supported(h, a) ? direct_time(h, a) : 1e30, slab = a.conv ? 1e30 : slab_time(h, a);
  const Plan pl = plan_for(h, a);
  const double keep = (double)h->nnz / (double)h->M, per = pl.whole ? (double)h->sp_ktiles : (double)pl.kt_per;
  const double threads = slab < direct ? slab_parts(h, a) : direct_parts(h, a), more = threads > 1.0 ? threads : 0.0;
  const double share = per / (pl.whole ? 1.0 : (double)pl.parts);
  const double here = a.conv ? 3.4e-15 + 2.5e-16 * per : 4.9e-15 + 2.1e-16 * per;
  const double there = (a.conv ? 1.69e-16 : 2.89e-16) * keep / threads + 4.8e-16 * more;
  const double here1 = a.conv ? 2.8e-15 + 1.3e-16 * share : 3.4e-15 + 1.2e-16 * share;
  const double there1 = a.conv ? 1.0e-15 + 0.9e-16 * keep / (threads * threads) + 2e-16 * more : 1.4e-15 + 2.2e-16 * keep / (threads * threads) + 2e-16 * more;
  return here <= there && here1 <= std::max(there1, 3.55e-15);
}

// Measured against the kernel that runs otherwise (us): 8192^2, 8 x 32, N = 1024: 665 -> 524 (593 at the power limit); 4096^2, 4 x 16, N = 512: 312 -> 91; 2880^2,
// 4 x 16, N = 17: 66 -> 24; 4096 x 512, rate 4, N = 512: 34 -> 20; 4096^2, 16 x 64, N = 1024: equal; 512 -> 512 channels, 28 x 28, one
// image: 62 -> 39.  Small matrices, few columns: 1533 x 2050, N = 131: 10.7 against 20, and so on.
// (Below ten million products the direct kernel is done before this one has filled its pipeline, some 12 us: no estimates for the
// smallest calls, 256^2, N = 64, whose 3.6 us are the host's: 3.65 -> 3.63.)
bool split_preferred(const grim_bcr* h, const SpmmArgs& a) {
  if (h->nnz * a.ncols < 10000000) return false;
  if (a.ncols <= kSkinnyMaxN || a.tile_n != 0 || (!a.conv && a.x_sq != 1) || !split_path_supported(h, a)) return false;
  const double direct = direct_path_supported(h, a) ? direct_time(h, a) : 1e30, slab = a.conv ? 1e30 : slab_time(h, a);
  return split_time(h, a) <= 0.92 * std::min(direct, slab) && split_precise(h, a);
}

grim_status_t launch_split(const grim_bcr* h, const SpmmArgs& a, cudaStream_t s) {
  if (!split_path_supported(h, a)) return GRIM_ERR_UNSUPPORTED;
  SplitParams p;
  p.w.head = h->d_rc_head; p.w.blob = h->d_rc_blob; p.w.nbc = (int)h->nbc; p.w.bw = h->bw;
  p.stage = h->d_sp_stage; p.blob = h->d_sp_blob; p.band_order = h->d_band_order; p.status = h->d_status;
  p.nbr = (int)h->nbr; p.M = (int)h->M; p.K = (int)h->K; p.nbc = (int)h->nbc;
  p.nkt = (int)h->sp_ktiles;
  p.mtiles = (int)h->sp_mtiles;
  CUtensorMap tm = {};
  p.tma = rows_by_tma(h, a) && matrix_map_f32(a.X, a.ncols, h->K, a.x_sk, kTile, kK, &tm);
  p.nrec = rec_slots(h, p.tma);
  p.rec_stride = rec_stride_of(h);
  p.spin_limit = 1u << 20;
  p.a = a;
  Plan pl = plan_for(h, a);
  const int asked = a.tile_n - 64;  // test / tuning override
  if (asked > 0 && asked <= kMaxParts && (asked - 1) * ((p.nkt + asked - 1) / asked) < p.nkt)
    pl = {0, pl.whole + pl.tail, asked, (p.nkt + asked - 1) / asked};
  if (pl.parts == 1) pl = {0, pl.whole + pl.tail, 1, p.nkt};
  const size_t smem = smem_need(h, p.nrec, p.tma);
  auto launch = [&](int64_t first, int64_t tiles, int parts, int kt_per) {
    p.tile0 = (int)first;
    p.parts = parts;
    p.kt_per = kt_per;
    const unsigned grid = (unsigned)(tiles * parts);
    count_launch();
    return h->bh == 4 ? launch_rows<4>(tm, p, grid, smem, s) : (h->bh == 8 ? launch_rows<8>(tm, p, grid, smem, s) : launch_rows<16>(tm, p, grid, smem, s));
  };
  cudaError_t e = cudaSuccess;
  if (pl.whole) e = launch(0, pl.whole, 1, p.nkt);
  if (pl.tail && e == cudaSuccess) e = launch(pl.whole, pl.tail, pl.parts, pl.kt_per);
  if (e != cudaSuccess) { cudaGetLastError(); return GRIM_ERR_CUDA; }
  return GRIM_OK;
}

}  // namespace grim
