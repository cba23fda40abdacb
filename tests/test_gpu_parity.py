"""GPU parity: every CUDA entry point against the fp64 CPU oracle, element by element, through the C ABI.

Tolerances (fixed requirements of this library): fp32 results  ||Y - Y*||_F / ||Y*||_F <= 1e-5;
bf16 inputs with fp32 accumulation  max |err| <= 2e-2 * ||W row||_2 * ||X col||_2 (plus |bias| where
a bias is added); packing is bit-exact (tests/test_packer_host.py).  Rows kept by no block must be
exactly +0.
"""
import numpy as np
import pytest
import torch

from oracle import bcr_oracle as orc
from parity_util import F32_TOL, assert_close, rel_fro
from workloads import generators as gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2108_11033_b200.build import build_library
    build_library()
    from paper_2108_11033_b200 import binding
    return binding


def to_dev(a, bf16=False):
    t = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    return t.to(torch.bfloat16) if bf16 else t


def check_spmm(B, W, mask, X, bh, bw, *, bf16=False, flags=0, tile_n=0, y_bf16=False, path=0):
    M, K = W.shape
    X = gen.bf16_representable(X) if bf16 else np.asarray(X, np.float32)
    N = X.shape[1]
    dt = B.GRIM_BF16 if bf16 else B.GRIM_F32
    h = B.grim_bcr_pack(W, mask, bh, bw, dt, flags)
    try:
        if bf16:
            B.grim_bcr_reserve(h, N)  # workspace of the split tensor-core multiply, where the library chooses it
        Xd = to_dev(X, bf16)
        Yd = torch.full((M, N), float("nan"), device="cuda", dtype=torch.bfloat16 if y_bf16 else torch.float32)
        if tile_n or path:
            B.grim_bcr_spmm_ex(h, Xd, Yd, tile_n=tile_n, path=path)
        else:
            B.grim_bcr_spmm(h, Xd, Yd)
        torch.cuda.synchronize()
        assert B.grim_bcr_status(h) == B.GRIM_OK
        got = Yd.float().cpu().numpy().astype(np.float64)
        want = orc.spmm(W, mask, X, dt)
        dead = np.flatnonzero(mask.sum(axis=1) == 0)
        assert np.all(got[dead] == 0.0) and not np.any(np.signbit(got[dead])), "pruned rows must be exactly +0"
        Wm = orc.masked_weight(W, mask, dt)
        scale = np.linalg.norm(Wm, axis=1)[:, None] * np.linalg.norm(X.astype(np.float64), axis=0)[None, :]
        assert_close(got, want, scale, bf16_in=bf16, out_bf16=y_bf16, what=f"spmm {M}x{K}x{N}")
    finally:
        B.grim_bcr_destroy(h)


# ---------------------------------------------------------------------------------------- SpMM / GEMV


def test_config1_spmm_fp32(B):
    c = gen.config1_spmm()
    check_spmm(B, c["W"], c["mask"], c["X"], c["bh"], c["bw"])


SHAPES = [
    # M, K, bh, bw, generator kwargs
    (256, 256, 16, 16, dict(dist="fixed", kr_fixed=8, kc_fixed=8)),
    (200, 333, 8, 32, dict(compression=6, dist="uniform")),
    (96, 153, 8, 32, dict(compression=10, dist="uniform")),
    (130, 260, 4, 16, dict(compression=8, dist="zipf")),
    (150, 500, 16, 64, dict(compression=4, dist="zipf", empty_frac=0.25)),
    (64, 27, 8, 32, dict(compression=3, dist="uniform")),
    (33, 40, 3, 5, dict(compression=2, dist="uniform")),
    (24, 48, 1, 1, dict(compression=3, dist="uniform")),
    (16, 64, 16, 64, dict(compression=4, dist="uniform")),
]


@pytest.mark.parametrize("N", [1, 3, 16, 37, 64, 130, 260])
@pytest.mark.parametrize("shape", SHAPES)
def test_spmm_fp32_small(B, shape, N):
    M, K, bh, bw, kw = shape
    W = gen.dense_weight(M, K, seed=60)
    mask = gen.bcr_mask(M, K, bh, bw, seed=61, **kw)
    X = gen.normal_f32((K, N), 1.0, 62, 0)
    check_spmm(B, W, mask, X, bh, bw)


@pytest.mark.parametrize("N", [1, 5, 64, 200])
@pytest.mark.parametrize("shape", SHAPES[1:6])
def test_spmm_bf16_small(B, shape, N):
    M, K, bh, bw, kw = shape
    W = gen.dense_weight(M, K, seed=63)
    mask = gen.bcr_mask(M, K, bh, bw, seed=64, **kw)
    X = gen.normal_f32((K, N), 1.0, 65, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=True)
    check_spmm(B, W, mask, X, bh, bw, bf16=True, y_bf16=True)


@pytest.mark.parametrize("tile_n", [16, 32, 64, 128])
@pytest.mark.parametrize("reorder", [0, 1])
def test_spmm_tiles_and_reorder(B, tile_n, reorder):
    M, K, bh, bw = 512, 768, 8, 32
    W = gen.dense_weight(M, K, seed=66)
    mask = gen.bcr_mask(M, K, bh, bw, compression=8, dist="zipf", seed=67, empty_frac=0.1)
    mask[40:56] = 0  # two fully pruned bands
    X = gen.normal_f32((K, 150), 1.0, 68, 0)
    check_spmm(B, W, mask, X, bh, bw, flags=reorder, tile_n=tile_n)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", [(512, 768, 8, 32, 1), (512, 768, 8, 32, 2), (300, 520, 4, 16, 4), (300, 520, 4, 16, 1),
                                  (260, 700, 16, 64, 1), (96, 153, 8, 32, 2), (64, 27, 8, 32, 1), (33, 40, 3, 5, 1)])
def test_register_tiled_kernel_explicit(B, case, bf16):
    """The N > 16 register-tiled kernel asked for by name (path 1), with each number of band groups per
    thread block, on a ragged column count (TMA loader: aligned X; gather loader: covered by the strided test)."""
    M, K, bh, bw, groups = case
    W = gen.dense_weight(M, K, seed=73)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=74, empty_frac=0.1)
    mask[: 2 * bh] = 0
    X = gen.normal_f32((K, 328), 1.0, 75, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=bf16, tile_n=groups, path=1, flags=1)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", [(512, 768, 8, 32, 8, 328), (512, 768, 8, 32, 8, 600), (300, 520, 4, 16, 8, 328),
                                  (300, 520, 4, 16, 9, 515), (96, 153, 8, 32, 8, 257), (64, 27, 8, 32, 8, 1024)])
def test_register_tiled_kernel_two_pieces_per_lane(B, case, bf16):
    """The same kernel with 256-column tiles (a lane owns two 4-column pieces; tile_n 8 and 9), on column counts that
    leave the second piece partly or wholly empty in the last tile."""
    M, K, bh, bw, tile_n, N = case
    W = gen.dense_weight(M, K, seed=173)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=174, empty_frac=0.1)
    mask[: 2 * bh] = 0
    X = gen.normal_f32((K, N), 1.0, 175, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=bf16, tile_n=tile_n, path=1, flags=1)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", [(512, 768, 8, 32, 17, 16), (512, 768, 8, 32, 18, 12), (512, 768, 8, 32, 20, 9),
                                  (300, 520, 4, 16, 20, 16), (260, 700, 16, 64, 17, 16), (96, 153, 8, 32, 17, 5),
                                  (64, 27, 8, 32, 17, 1), (2048, 1024, 8, 32, 17 + 256 * 3, 16)])
def test_register_tiled_kernel_narrow_tile(B, case, bf16):
    """The 16-column tile for N <= 16 (a lane owns one column, the halves of a warp split each chunk's kept columns;
    tile_n 17, 18, 20 = 1, 2, 4 band groups per thread block), unsplit and split over the block columns."""
    M, K, bh, bw, tile_n, N = case
    W = gen.dense_weight(M, K, seed=183)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=184, empty_frac=0.1)
    mask[: 2 * bh] = 0
    X = gen.normal_f32((K, N), 1.0, 185, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=bf16, tile_n=tile_n, path=1, flags=1)


@pytest.mark.parametrize("row_tiles", [1, 2])
def test_tensor_core_row_tiles_per_block(B, row_tiles):
    """One or two 128-row tiles per thread block (two share every X tile), on a row count that leaves the last
    thread block with a single, partly filled tile."""
    M, K, bh, bw, N = 328, 700, 8, 32, 520
    W = gen.dense_weight(M, K, seed=97)
    mask = gen.bcr_mask(M, K, bh, bw, compression=5, dist="uniform", seed=98, empty_frac=0.1)
    X = gen.normal_f32((K, N), 1.0, 99, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=True, path=2, tile_n=row_tiles, flags=1)


@pytest.mark.parametrize("y_bf16", [False, True])
@pytest.mark.parametrize("case", [(256, 512, 8, 32, 256), (200, 333, 8, 32, 328), (300, 520, 4, 16, 520), (260, 700, 16, 64, 264),
                                  (96, 153, 8, 32, 1024), (512, 2048, 16, 64, 776)])
def test_tensor_core_kernel_explicit(B, case, y_bf16):
    """The tcgen05 path asked for by name (path 2): bf16 operands, fp32 accumulation in tensor memory; ragged M, K
    and N, empty blocks, pruned bands, every supported block shape."""
    M, K, bh, bw, N = case
    W = gen.dense_weight(M, K, seed=87)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=88, empty_frac=0.1)
    mask[: 2 * bh] = 0
    X = gen.normal_f32((K, N), 1.0, 89, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=True, path=2, flags=1, y_bf16=y_bf16)


@pytest.mark.parametrize("y_bf16", [False, True])
@pytest.mark.parametrize("case", [(256, 512, 8, 32, 512), (328, 700, 8, 32, 520), (300, 520, 4, 16, 1032), (260, 700, 16, 64, 264),
                                  (96, 153, 8, 32, 1024), (512, 2048, 16, 64, 776), (640, 320, 4, 32, 600), (400, 256, 8, 16, 520),
                                  (384, 448, 16, 16, 512), (384, 448, 16, 32, 136), (200, 333, 4, 64, 328), (1100, 900, 8, 64, 1544)])
def test_paired_tensor_core_kernel_explicit(B, case, y_bf16):
    """The paired tcgen05 kernel asked for by name (path 5): two thread blocks multiply 256 rows x 512 columns
    together.  Ragged M, K and N, an odd number of 128-row tiles (the last pair has one empty partner), a single
    tile, empty blocks, pruned bands, every supported block shape."""
    M, K, bh, bw, N = case
    W = gen.dense_weight(M, K, seed=187)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=188, empty_frac=0.1)
    mask[: 2 * bh] = 0
    X = gen.normal_f32((K, N), 1.0, 189, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=True, path=5, flags=1, y_bf16=y_bf16)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", [(304, 520, 4, 16, 1, 1, 31), (300, 700, 8, 32, 1, 16, 33), (129, 333, 16, 64, 2, 16, 63),
                                  (300, 520, 4, 16, 2, 4, 65), (260, 700, 16, 64, 4, 8, 131), (512, 768, 8, 32, 4, 2, 256),
                                  (200, 300, 5, 20, 4, 1, 129), (7, 40, 3, 9, 2, 8, 5), (512, 2100, 8, 32, 2, 8, 130), (96, 96, 16, 16, 1, 2, 2)])
def test_direct_kernel_explicit(B, case, bf16):
    """Columns per lane x warps per band: widths around a tile's edge, vector and scalar loads of X, bands with nothing
    kept, block sizes below the compiled row counts, more warps per band than block columns."""
    M, K, bh, bw, nc, parts, N = case
    W = gen.dense_weight(M, K, seed=171)
    mask = gen.bcr_mask(M, K, bh, bw, compression=3, dist="zipf", seed=172, empty_frac=0.3)
    mask[:bh] = 0
    X = gen.normal_f32((K, N), 1.0, 173, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=bf16, path=1, tile_n=32 + nc + 256 * parts, y_bf16=bf16 and parts == 1)


@pytest.mark.parametrize("bf16", [False, True])
def test_more_bands_than_the_direct_kernel_takes(B, bf16):
    """Half a million rows in blocks of one row, rows of X that TMA cannot fetch: the other CUDA-core kernels take them."""
    M, K, N = 524288 + 24, 32, 17
    W = gen.normal_f32((M, K), 1.0, 178, 0)
    mask = (gen.normal_f32((M, K), 1.0, 179, 0) > 0.7).astype(np.uint8)
    X = gen.normal_f32((K, N), 1.0, 180, 0)
    if bf16:
        W, X = gen.bf16_representable(W), gen.bf16_representable(X)
    h = B.grim_bcr_pack(W, mask, 1, 32, B.GRIM_BF16 if bf16 else B.GRIM_F32, 0)
    try:
        Y = torch.full((M, N), float("nan"), device="cuda")
        B.grim_bcr_spmm(h, to_dev(X, bf16), Y)
        assert rel_fro(Y.cpu().numpy(), (W * mask).astype(np.float64) @ X.astype(np.float64)) <= F32_TOL
    finally:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("geom", [(3, 1, 1, 9, 13), (3, 2, 1, 15, 8), (5, 1, 2, 7, 7), (1, 2, 0, 9, 9), (16, 3, 5, 21, 19), (2, 1, 0, 6, 33)])
def test_direct_kernel_convolution(B, geom, bf16):
    ksize, stride, pad, hh, ww = geom
    W = gen.dense_weight(40, 6 * ksize * ksize, seed=174)
    mask = gen.bcr_mask(40, 6 * ksize * ksize, 8, 32, compression=3, dist="uniform", seed=175, empty_frac=0.2)
    x = np.maximum(gen.normal_f32((3, 6, hh, ww), 1.0, 176, 0), 0.0)
    L = dict(W=W, mask=mask, bias=gen.normal_f32((40,), 0.05, 177, 0), bh=8, bw=32)
    check_conv(B, L, x, ksize=ksize, stride=stride, pad=pad, bf16=bf16, kernel_flags=B.GRIM_CONV_DIRECT)


def split_and_direct(B, W, mask, X, bh, bw, parts, flags=0):
    """Results of the kernel that splits operands and of the direct kernel, which have to be two kernels."""
    h = B.grim_bcr_pack(W, mask, bh, bw, B.GRIM_F32, flags)
    try:
        out = []
        for tile_n in (64 + parts, 32):
            Y = torch.full((W.shape[0], X.shape[1]), 7.0, device="cuda")
            B.grim_bcr_spmm_ex(h, to_dev(X), Y, path=1, tile_n=tile_n)
            out.append(Y.cpu().numpy())
        assert B.grim_bcr_status(h) == B.GRIM_OK
    finally:
        B.grim_bcr_destroy(h)
    assert not np.array_equal(out[0], out[1], equal_nan=True)
    return out


@pytest.mark.parametrize("parts", [1, 2, 3, 8])
@pytest.mark.parametrize("case", [(128, 512, 128, 8, 32), (130, 1000, 129, 8, 16), (259, 1500, 30, 16, 64), (600, 1000, 260, 4, 16), (33, 1500, 17, 4, 64), (300, 990, 1, 16, 16)])
def test_split_operands(B, case, parts):
    """Operands as three bf16 numbers each: rows, columns and K just past the tiles of 128, 128 and 64, every block height, up to eight
    thread blocks to a tile (the last with less of K; eight share 8, 16 and 24 K tiles); rows and bands that keep nothing."""
    M, K, N, bh, bw = case
    W = gen.dense_weight(M, K, seed=411)
    mask = gen.bcr_mask(M, K, bh, bw, compression=5, dist="zipf", seed=412, empty_frac=0.15)
    mask[:2 * bh] = 0
    X = gen.normal_f32((K, N), 1.0, 413, 0)
    X[::3] = np.maximum(X[::3], 0.0)
    check_spmm(B, W, mask, X, bh, bw, flags=parts & 1, path=1, tile_n=64 + parts)
    split_and_direct(B, W, mask, X, bh, bw, parts, parts & 1)


@pytest.mark.parametrize("M,K,N", [(1300, 1000, 1810), (390, 1100, 4900), (2600, 520, 1800)])
def test_split_operands_last_round(B, M, K, N):
    """More tiles than SMs: whole rounds in one launch, the tiles of the last one shared by clusters in another (165 tiles: 17 by eight
    blocks; 156: 8; 315: 19, of a K that is cut into fewer parts than that)."""
    W = gen.dense_weight(M, K, seed=441)
    mask = gen.bcr_mask(M, K, 8, 32, compression=6, dist="uniform", seed=442)
    X = gen.normal_f32((K, N), 1.0, 443, 0)
    check_spmm(B, W, mask, X, 8, 32, path=1, tile_n=64)
    split_and_direct(B, W, mask, X, 8, 32, 0)


# Per element, against what the row itself keeps: fp32 sums lose about eps32 * sqrt(sum of squared products), times the square
# root of the number of additions (below 700); the 64-fold covers both and what the split leaves out (2^-25 of every product).
# (times: a longer sum's square root beside that of 700 additions)
def assert_elements(got, Wm, X, times=1):
    Wm, X = Wm.astype(np.float64), X.astype(np.float64)
    scale = np.sqrt((Wm ** 2) @ (X ** 2))
    assert np.all(np.abs(got - Wm @ X) <= 64 * times * 2.0 ** -24 * scale + 1e-44)


@pytest.mark.parametrize("parts", [1, 3])
@pytest.mark.parametrize("bh,bw,K", [(4, 16, 700), (8, 32, 700), (16, 64, 700), (8, 32, 16500)])
def test_split_operands_of_any_range(B, bh, bw, K, parts):
    """Rows of very different size; and columns of X that are not split - an infinity, a NaN, numbers near the ends of fp32's range -
    are as good as the others, and nothing of them reaches a row that does not keep them or another column.  (16500: more K tiles to a
    thread block than have flags of their own.)"""
    M, N = 300, 140
    W = gen.dense_weight(M, K, seed=421)
    W[np.abs(W) < 1e-3] = 0.01
    mask = gen.bcr_mask(M, K, bh, bw, compression=4, dist="uniform", seed=422, empty_frac=0.2)
    X = gen.normal_f32((K, N), 1.0, 423, 0)
    used = np.flatnonzero(mask.any(axis=0))
    X[:, 3] *= 10.0 ** (np.arange(K) % 13 - 6)
    X[:, 40] *= np.float32(1e-36)
    X[:, 41] *= np.float32(1e35)
    X[:, 42] = 0.0
    X[:, 43] *= np.where(np.arange(K) % 16 == 0, 1.0, 1e-7).astype(np.float32)
    X[:, 44] *= np.float32(2.0 ** -107)  # some below what is split, most above
    X[:, 45] *= np.float32(2.0 ** 61)
    X[used[5], 128], X[used[40], 129], X[used[-1], 139] = np.inf, np.nan, -np.inf
    got, _ = split_and_direct(B, W, mask, X, bh, bw, parts)
    fin = np.isfinite(X)
    X0, Wm = np.where(fin, X, 0.0).astype(np.float64), (W * mask).astype(np.float64)
    want = Wm @ X0
    for k, q in zip(*np.nonzero(~fin)):
        want[mask[:, k] != 0, q] += W[mask[:, k] != 0, k].astype(np.float64) * X[k, q]
    ok = np.isfinite(want)
    assert not ok.all() and np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    assert_elements(np.where(ok, got, Wm @ X0), Wm, X0, 4 if K > 700 else 1)


@pytest.mark.parametrize("parts", [1, 3])
@pytest.mark.parametrize("large", ["activations", "weights"])
@pytest.mark.parametrize("few", [1, 2, 24])
@pytest.mark.parametrize("power", [17, 20, 24, 28, 36, 40, 60])
def test_split_operands_elements_beside_large_ones(B, power, few, large, parts):
    """In every 64 of k one activation that is 2^power times the others, in every row weights that are; one, two or many others.  A row
    that keeps none of the large activations, a column that is zero at the large weights, consists of the others alone: its
    elements are as exact as any."""
    M, K, N, bh, bw = 320, 512, 136, 8, 32
    W = gen.dense_weight(M, K, seed=451)
    W[np.abs(W) < 1e-3] = 0.01
    mask = gen.bcr_mask(M, K, bh, bw, compression=5, dist="uniform", seed=452)
    rng = np.random.default_rng(453)
    keep = rng.random((K // 64, 64, N)).argsort(axis=1).reshape(K, N) < few
    X = np.where(keep, gen.normal_f32((K, N), 1.0, 454, 0), np.float32(0))
    at = np.arange(K // 64) * 64 + 1 + 7 * np.arange(K // 64)
    if large == "activations":
        X[at] = np.float32(1.3 * 2.0 ** power)
        small = (mask[:, at] == 0).all(axis=1)  # rows
        assert 5 < small.sum() < M - 5
    else:
        others = np.setdiff1d(np.arange(K), at[:few]) if few <= 2 else at
        W[:, others] *= np.float32(2.0 ** (power - 30))
        W[:, np.setdiff1d(np.arange(K), others)] *= np.float32(2.0 ** -30)
        X[at[:few]] = 1.0
        X[others, : N // 2] = 0.0
    got, _ = split_and_direct(B, W, mask, X, bh, bw, parts)
    assert_elements(got, W * mask, X)


@pytest.mark.parametrize("M,K,rate,N", [(1024, 1024, 8, 640), (2048, 512, 16, 640), (2048, 512, 16, 768)])
def test_tuned_split_operands_only_where_as_exact(B, M, K, rate, N):
    """The tile search at 1024 columns finds the kernel above; at widths of the same power of two where that is less exact than what runs
    otherwise, the search's answer is not taken."""
    W = gen.dense_weight(M, K, seed=471)
    mask = gen.bcr_mask(M, K, 4, 16, compression=rate, dist="uniform", seed=472)
    X = to_dev(gen.normal_f32((K, 1024), 1.0, 473, 0))
    tuned, plain = (B.grim_bcr_pack(W, mask, 4, 16, B.GRIM_F32, 1) for _ in range(2))
    try:
        t = B.grim_bcr_tune(tuned, X, torch.empty(M, 1024, device="cuda"), reps=20)
        if (t["path"], t["tile_n"]) != (1, 64):  # (it takes 20 us here and the next one 27)
            pytest.skip("another kernel was faster")
        out = []
        for h in (tuned, plain):
            out.append(torch.empty(M, N, device="cuda"))
            B.grim_bcr_spmm(h, X[:, :N].contiguous(), out[-1])
        assert torch.equal(*out)
    finally:
        B.grim_bcr_destroy(tuned)
        B.grim_bcr_destroy(plain)


def test_tile_search_at_sixteen_columns_leaves_split_operands_out(B):
    """There the kernels that run otherwise spread a row over 32 lanes and are more exact."""
    M = K = 8192
    h = B.grim_bcr_pack(gen.dense_weight(M, K, seed=474), gen.bcr_mask(M, K, 8, 32, compression=4, dist="uniform", seed=475), 8, 32, B.GRIM_F32, 1)
    try:
        X = to_dev(gen.normal_f32((K, 16), 1.0, 476, 0))
        t = B.grim_bcr_tune(h, X, torch.empty(M, 16, device="cuda"), reps=-3)
        assert (t["path"], t["tile_n"]) != (1, 64)
    finally:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("geom", [(1, 200, 130, 25, 27, 3, 1, 1), (2, 133, 260, 31, 33, 5, 2, 2), (3, 400, 72, 61, 63, 3, 2, 0),
                                  (3, 16, 264, 48, 61, 16, 3, 5), (2, 700, 500, 30, 29, 1, 1, 0), (5, 400, 520, 13, 15, 3, 1, 1)])
def test_split_operands_convolution(B, geom):
    """Convolutions that the kernel above is preferred for: pixels and rows just past its tiles, tiles that meet two images, strides,
    kernels of 1 to 16; one thread block to a tile and several."""
    nb, cin, cout, hh, ww, ksize, stride, pad = geom
    K = cin * ksize * ksize
    mask = gen.bcr_mask(cout, K, 8, 32, compression=3, dist="uniform", seed=431, empty_frac=0.1)
    x = np.maximum(gen.normal_f32((nb, cin, hh, ww), 1.0, 432, 0), 0.0)
    L = dict(W=gen.dense_weight(cout, K, seed=433), mask=mask, bias=gen.normal_f32((cout,), 0.05, 434, 0), bh=8, bw=32)
    y = check_conv(B, L, x, ksize=ksize, stride=stride, pad=pad, bf16=False)
    direct = check_conv(B, L, x, ksize=ksize, stride=stride, pad=pad, bf16=False, kernel_flags=B.GRIM_CONV_DIRECT)
    assert not np.array_equal(y, direct)  # (another kernel)


@pytest.mark.parametrize("out_bf16", [False, True])
@pytest.mark.parametrize("geom", [
    (1, 64, 64, 16, 16, 3, 1, 1), (2, 30, 72, 9, 13, 3, 1, 1), (2, 17, 48, 12, 10, 5, 2, 2), (1, 130, 300, 15, 17, 3, 2, 1),
    (3, 96, 136, 14, 14, 3, 1, 0), (1, 512, 256, 7, 7, 3, 1, 1), (40, 40, 264, 30, 31, 3, 1, 1), (24, 64, 512, 28, 28, 3, 1, 1),
    (2, 3, 40, 20, 24, 3, 1, 1), (3, 2, 70, 19, 23, 5, 2, 2), (1, 64, 24, 9, 9, 1, 2, 0), (1, 1, 16, 21, 13, 8, 3, 4)])
def test_tensor_core_convolution(B, geom, out_bf16):
    """Channel-last kernel: 16, 32 and 64 channels per copy, ragged channels, pixels and planes of odd size, several tiles per
    thread block, pairs of blocks, K split over a cluster, stride and padding; and the gathering variant (K <= 64)."""
    nb, cin, cout, hh, ww, ksize, stride, pad = geom
    K = cin * ksize * ksize
    W = gen.dense_weight(cout, K, seed=181)
    mask = gen.bcr_mask(cout, K, 8, 32, compression=3, dist="uniform", seed=182, empty_frac=0.2)
    mask[:8] = 0
    x = np.maximum(gen.normal_f32((nb, cin, hh, ww), 1.0, 183, 0), 0.0)
    L = dict(W=W, mask=mask, bias=gen.normal_f32((cout,), 0.05, 184, 0), bh=8, bw=32)
    check_conv(B, L, x, ksize=ksize, stride=stride, pad=pad, bf16=True, out_bf16=out_bf16, kernel_flags=B.GRIM_CONV_TENSOR)


@pytest.mark.parametrize("cin", [3, 16])
def test_convolution_bias_from_the_call_before(B, cin):
    """The biases are the result of a product issued just before on the same stream (few long bands: it runs long after its
    launch has let the next one start); with and without the channel-last launch in between.  Bit for bit what the
    convolution gives when the product has long been done."""
    cout, Kb = 40, 60000
    hb = B.grim_bcr_pack(gen.dense_weight(cout, Kb, seed=188), gen.bcr_mask(cout, Kb, 8, 32, compression=2, dist="uniform", seed=189), 8, 32, B.GRIM_F32, 0)
    K = cin * 9
    h = B.grim_bcr_pack(gen.dense_weight(cout, K, seed=190), gen.bcr_mask(cout, K, 8, 32, compression=3, dist="uniform", seed=191), 8, 32, B.GRIM_BF16, 0)
    try:
        xb = to_dev(gen.normal_f32((Kb, 1), 1.0, 192, 0))
        x = to_dev(gen.normal_f32((2, cin, 20, 24), 1.0, 193, 0), True)
        B.grim_bcr_reserve(h, 2 * 20 * 24)
        bias, out, want = torch.empty(cout, 1, device="cuda"), torch.empty(2, cout, 20, 24, device="cuda"), torch.empty(2, cout, 20, 24, device="cuda")
        B.grim_bcr_spmm(hb, xb, bias)
        torch.cuda.synchronize()
        B.grim_bcr_conv2d(h, x, want, 3, 1, 1, bias=bias, kernel_flags=B.GRIM_CONV_TENSOR)
        for _ in range(20):
            bias.fill_(1e6)
            torch.cuda.synchronize()
            B.grim_bcr_spmm(hb, xb, bias)
            B.grim_bcr_conv2d(h, x, out, 3, 1, 1, bias=bias, kernel_flags=B.GRIM_CONV_TENSOR)
            assert torch.equal(out, want)
    finally:
        B.grim_bcr_destroy(h)
        B.grim_bcr_destroy(hb)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("hw", [(6, 10), (4, 8), (2, 24), (10, 16), (8, 32)])
def test_maxpool_vector_widths(B, bf16, hw):
    """Output rows of 5, 4, 12, 8 and 16 elements: scalar passes and vectors of 2, 4 and 8; exact."""
    x = to_dev(gen.normal_f32((3, 5) + hw, 1.0, 185, 0), bf16)
    out = torch.empty(3, 5, hw[0] // 2, hw[1] // 2, device="cuda", dtype=x.dtype)
    B.grim_maxpool2x2(x, out)
    assert torch.equal(out, torch.nn.functional.max_pool2d(x, 2))


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("parts", [1, 2, 4, 8])
@pytest.mark.parametrize("case", [(300, 700, 8, 32, 2), (304, 520, 4, 16, 3), (129, 1333, 16, 64, 4), (300, 520, 4, 16, 7), (512, 2100, 8, 32, 8),
                                  (260, 700, 16, 64, 9), (200, 300, 5, 20, 12), (7, 40, 3, 9, 15), (520, 1040, 8, 32, 16), (264, 512, 4, 16, 16)])
def test_gathering_kernel(B, case, parts, bf16):
    """One to several passes over the columns, rows of X with and without aligned pieces, bands with fewer chunks than warps
    or none, short last chunks, block heights below the compiled ones."""
    M, K, bh, bw, N = case
    W = gen.dense_weight(M, K, seed=191)
    mask = gen.bcr_mask(M, K, bh, bw, compression=4, dist="zipf", seed=192, empty_frac=0.3)
    mask[:bh] = 0
    X = gen.normal_f32((K, N), 1.0, 193, 0)
    check_spmm(B, W, mask, X, bh, bw, bf16=bf16, path=3, tile_n=8 * parts, y_bf16=bf16 and parts == 2)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", [(300, 700, 8, 32, 1), (300, 700, 8, 32, 3), (300, 700, 8, 32, 5), (304, 520, 4, 16, 7), (260, 700, 16, 64, 2), (260, 700, 16, 64, 6),
                                  (129, 1333, 16, 64, 12), (520, 1040, 8, 32, 16), (304, 520, 4, 16, 16), (264, 700, 8, 32, 11), (2048, 2048, 8, 32, 6), (200, 300, 5, 20, 8)])
def test_non_finite_activations_reach_only_rows_that_keep_them(B, case, bf16):
    """At most sixteen columns: infinities and a NaN in X meet the rows whose weight at their column is kept, and no other."""
    M, K, bh, bw, N = case
    W = gen.dense_weight(M, K, seed=311)
    W[np.abs(W) < 1e-3] = 0.01  # (a kept weight of zero would make a NaN of an infinity)
    mask = gen.bcr_mask(M, K, bh, bw, compression=4, dist="zipf", seed=312, empty_frac=0.2)
    mask[:bh] = 0
    X = gen.normal_f32((K, N), 1.0, 313, 0)
    X = gen.bf16_representable(X) if bf16 else X
    used = np.flatnonzero(mask.any(axis=0))
    X[used[3], 0], X[used[len(used) // 2], N // 2], X[used[-1], N - 1] = np.inf, -np.inf, np.nan
    Wd = gen.bf16_representable(W) if bf16 else W
    h = B.grim_bcr_pack(W, mask, bh, bw, B.GRIM_BF16 if bf16 else B.GRIM_F32, 0)
    try:
        Yd = torch.full((M, N), 7.0, device="cuda")
        B.grim_bcr_spmm(h, to_dev(X, bf16), Yd)
        got = Yd.cpu().numpy()
    finally:
        B.grim_bcr_destroy(h)
    fin = np.isfinite(X)
    want = (Wd * mask).astype(np.float64) @ np.where(fin, X, 0.0).astype(np.float64)
    for k, q in zip(*np.nonzero(~fin)):
        rows = mask[:, k] != 0
        with np.errstate(invalid="ignore"):
            want[rows, q] += Wd[rows, k].astype(np.float64) * X[k, q]
    bad = ~np.isfinite(want)
    assert bad.any() and not bad.all()
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    # finite results as ever: bf16 products are exact in fp32, sums of some hundred terms lose about sqrt(K) ulps of their terms
    scale = np.linalg.norm(Wd * mask, axis=1)[:, None] * np.linalg.norm(np.where(fin, X, 0.0), axis=0)[None, :]
    assert np.all(np.abs(got[~bad] - want[~bad]) <= 1e-5 * scale[~bad])


def test_handles_and_streams_in_other_forms(B):
    """A handle as a ctypes pointer; a stream as a torch stream, its address, or a number that is not a Python int."""
    import ctypes
    W, mask = gen.dense_weight(64, 96, seed=334), gen.bcr_mask(64, 96, 8, 32, compression=4, dist="uniform", seed=335)
    X = gen.normal_f32((96, 24), 1.0, 336, 0)
    h = B.grim_bcr_pack(W, mask, 8, 32, B.GRIM_F32, 0)
    try:
        want, Xd, s = (W * mask).astype(np.float64) @ X.astype(np.float64), to_dev(X), torch.cuda.Stream()
        for handle, stream in ((ctypes.c_void_p(h), None), (h, s), (h, s.cuda_stream), (h, np.int64(s.cuda_stream))):
            Y = torch.empty(64, 24, device="cuda")
            torch.cuda.synchronize()
            B.grim_bcr_spmm(handle, Xd, Y, stream)
            torch.cuda.synchronize()
            assert rel_fro(Y.cpu().numpy(), want) <= F32_TOL
        for handle, stream in ((2.5, None), ("h", None), (h, "s")):
            with pytest.raises((TypeError, ValueError)):
                B.grim_bcr_spmm(handle, Xd, Y, stream)
    finally:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("choice", [(1, 544, 40), (1, 33, 40), (1, 96, 40), (1, 128, 40), (1, 1056, 40), (3, 4, 1), (3, 8, 1), (3, 5, 7), (3, 12, 7), (3, 128, 7)])
def test_tile_values_without_a_meaning_run_the_default(B, choice):
    """Values of tile_n that name no tile of the path, or one for other widths."""
    path, tile_n, N = choice
    W, mask = gen.dense_weight(200, 520, seed=331), gen.bcr_mask(200, 520, 8, 32, compression=4, dist="uniform", seed=332)
    check_spmm(B, W, mask, gen.normal_f32((520, N), 1.0, 333, 0), 8, 32, path=path, tile_n=tile_n)


@pytest.mark.parametrize("case", [(300, 4, 16, False, 7, False), (300, 4, 16, False, 12, False), (300, 8, 32, False, 7, False), (300, 8, 32, False, 12, True),
                                  (300, 8, 32, True, 12, False), (1100, 8, 32, True, 16, True), (300, 8, 32, True, 17, True)])
def test_wide_handles_refuse_few_columns(B, case):
    """Handles with only the wide layouts: the widths, block heights and sizes that they refuse, and those that they take."""
    M, bh, bw, bf16, N, takes = case
    h = B.grim_bcr_pack(gen.dense_weight(M, 400, seed=328), gen.bcr_mask(M, 400, bh, bw, compression=8, dist="uniform", seed=329), bh, bw,
                        B.GRIM_BF16 if bf16 else B.GRIM_F32, B.GRIM_PACK_WIDE_ONLY)
    try:
        X, Y = torch.zeros(400, N, device="cuda", dtype=torch.bfloat16 if bf16 else torch.float32), torch.empty(M, N, device="cuda")
        if takes:
            B.grim_bcr_spmm(h, X, Y)
        else:
            with pytest.raises(B.GrimError) as e:
                B.grim_bcr_spmm(h, X, Y)
            assert e.value.status == B.GRIM_ERR_UNSUPPORTED
    finally:
        B.grim_bcr_destroy(h)


def test_reserve_of_more_columns_keeps_what_fewer_had(B):
    """An area for rows made aligned and one for the channel-last copy, whatever was reserved before or after: K x 7840 columns
    are more than the former may hold, 333 columns are not."""
    K = 512 * 9
    h = B.grim_bcr_pack(gen.dense_weight(128, K, seed=326), gen.bcr_mask(128, K, 8, 32, compression=8, dist="uniform", seed=327), 8, 32, B.GRIM_BF16, 0)
    try:
        X, Y = torch.zeros(K, 333, device="cuda", dtype=torch.bfloat16), torch.empty(128, 333, device="cuda")
        x, y = torch.zeros(10, 512, 28, 28, device="cuda", dtype=torch.bfloat16), torch.empty(10, 128, 28, 28, device="cuda")
        for ncols in ((7840,), (333, 7840), (7840, 333), (7840, 16)):
            B.grim_bcr_reserve(h, 0)
            for n in ncols:
                B.grim_bcr_reserve(h, n)
            B.grim_bcr_spmm_ex(h, X, Y, path=2)  # (refused where the rows cannot be copied)
            B.grim_bcr_conv2d(h, x, y, 3, 1, 1, kernel_flags=B.GRIM_CONV_TENSOR)
        torch.cuda.synchronize()
        assert B.grim_bcr_status(h) == 0 and not Y.any() and not y.any()
    finally:
        B.grim_bcr_destroy(h)


def test_reserve_stays_within_its_limit(B):
    """Few output channels, many input channels: M x max_ncols is within the limit, the channel-last copy would be 8 GiB."""
    K = 512 * 9
    h = B.grim_bcr_pack(gen.dense_weight(32, K, seed=324), gen.bcr_mask(32, K, 8, 32, compression=8, dist="uniform", seed=325), 8, 32, B.GRIM_BF16, 0)
    try:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        B.grim_bcr_reserve(h, (1 << 30) // (32 * 4))
        assert free - torch.cuda.mem_get_info()[0] <= (1 << 30) + (64 << 20)
        with pytest.raises(B.GrimError) as e:
            B.grim_bcr_reserve(h, (1 << 30) // (32 * 4) + 1)
        assert e.value.status == B.GRIM_ERR_UNSUPPORTED
    finally:
        B.grim_bcr_destroy(h)


def test_tuned_choice_that_cannot_take_the_operands(B):
    """Tuned on aligned rows (a tensor-core kernel wins); a product of the same kind whose rows start at odd elements, with no
    workspace to copy them to, runs all the same."""
    M, K, N = 2048, 2048, 512
    W, mask = gen.dense_weight(M, K, seed=321), gen.bcr_mask(M, K, 8, 32, compression=4, dist="uniform", seed=322)
    X = gen.bf16_representable(gen.normal_f32((K, N), 1.0, 323, 0))
    h = B.grim_bcr_pack(W, mask, 8, 32, B.GRIM_BF16, 0)
    try:
        Y = torch.empty(M, N, device="cuda")
        Xa = to_dev(X, True)
        assert B.grim_bcr_tune(h, Xa, Y)["path"] in (2, 5)
        Xu = torch.empty(K, N + 1, device="cuda", dtype=torch.bfloat16)[:, 1:]
        Xu.copy_(Xa)
        Y.fill_(float("nan"))
        B.grim_bcr_spmm(h, Xu, Y)
        assert rel_fro(Y.cpu().numpy(), (gen.bf16_representable(W) * mask).astype(np.float64) @ X.astype(np.float64)) <= F32_TOL
    finally:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("split", [2, 5, 8])
def test_split_multiply(B, split):
    """Few output tiles: several thread blocks share a tile's block columns and add their partial sums into a
    zeroed Y (pruned rows must stay exactly +0)."""
    M, K, bh, bw = 160, 2100, 8, 32
    W = gen.dense_weight(M, K, seed=83)
    mask = gen.bcr_mask(M, K, bh, bw, compression=8, dist="uniform", seed=84, empty_frac=0.2)
    mask[16:24] = 0
    X = gen.normal_f32((K, 200), 1.0, 85, 0)
    check_spmm(B, W, mask, X, bh, bw, path=1, tile_n=1 + 256 * split)


@pytest.mark.parametrize("case", [(2600, 330, 1100, 4, 16, 9), (5000, 400, 520, 8, 32, 8), (4800, 300, 1000, 16, 64, 1), (2500, 520, 260, 16, 32, 1)])
def test_slab_kernel_whole_and_split_tiles(B, case):
    """More tiles than SMs with few left over for the last round: whole tiles first, the rest shared by clusters in a second
    launch that starts before the first has ended.  Blocks whose last chunk is half padding or all of it in use."""
    M, K, N, bh, bw, tile = case
    W = gen.dense_weight(M, K, seed=87)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=88, empty_frac=0.2)
    X = gen.normal_f32((K, N), 1.0, 89, 0)
    check_spmm(B, W, mask, X, bh, bw, path=1, tile_n=tile)


@pytest.mark.parametrize("case", [(2300, 1030, 32, 8, 32), (2840, 1030, 30, 8, 32), (5630, 1025, 60, 16, 64), (2300, 1030, 12, 8, 32), (1000, 2050, 300, 4, 16)])
def test_slab_kernel_few_tiles(B, case):
    """Eighteen to thirty tiles, which clusters of five and six blocks share where the next size would take two rounds."""
    M, K, N, bh, bw = case
    W = gen.dense_weight(M, K, seed=85)
    mask = gen.bcr_mask(M, K, bh, bw, compression=8, dist="uniform", seed=84, empty_frac=0.2)
    check_spmm(B, W, mask, gen.normal_f32((K, N), 1.0, 83, 0), bh, bw, path=1, tile_n=17 if N <= 16 else 0)


@pytest.mark.parametrize("case", [(300, 5000, 24, 33, 1), (1100, 1300, 257, 257, 0), (700, 900, 40, 41, 3), (520, 1203, 1024, 1025, 2), (264, 6000, 17, 19, 0)])
@pytest.mark.parametrize("y_bf16", [False, True])
def test_tensor_core_rows_made_aligned(B, case, y_bf16):
    """bf16 right-hand sides whose rows TMA cannot fetch: copied to aligned rows (odd and even widths, rows that start inside a
    word, the last element of the buffer), outputs whose rows are not aligned either, with and without a split over K."""
    M, K, N, ld, off = case
    bh, bw = 8, 32
    W = gen.dense_weight(M, K, seed=301)
    mask = gen.bcr_mask(M, K, bh, bw, compression=2, dist="uniform", seed=302, empty_frac=0.1)
    X = gen.bf16_representable(gen.normal_f32((K, N), 1.0, 303, 0))
    flat = torch.full((off + (K - 1) * ld + N,), float("nan"), device="cuda", dtype=torch.bfloat16)
    Xd = torch.as_strided(flat, (K, N), (ld, 1), off)
    Xd.copy_(to_dev(X, True))
    h = B.grim_bcr_pack(W, mask, bh, bw, B.GRIM_BF16, 0)
    try:
        B.grim_bcr_reserve(h, N)
        Yd = torch.full((M, N), float("nan"), device="cuda", dtype=torch.bfloat16 if y_bf16 else torch.float32)
        B.grim_bcr_spmm(h, Xd, Yd)
        ref = (gen.bf16_representable(W) * mask).astype(np.float64) @ X.astype(np.float64)
        # bf16 products are exact in fp32; sums of a few thousand terms lose about sqrt(K) ulps, a bf16 result 2^-9
        assert rel_fro(Yd.float().cpu().numpy(), ref) <= (3e-3 if y_bf16 else 1e-5)
        assert B.grim_bcr_status(h) == 0
    finally:
        B.grim_bcr_destroy(h)


def test_conv_split_with_bias_and_relu(B):
    """A layer with few output pixels and many input channels takes the split path (separate bias / ReLU pass)."""
    L = gen.conv_layer(1, 96, 48, 9, ksize=3, bh=8, bw=32, compression=4, seed=86)
    check_conv(B, L, L["x"], ksize=3, stride=1, pad=1, bf16=False)
    check_conv(B, L, L["x"], ksize=3, stride=1, pad=1, bf16=False, relu=False)


@pytest.mark.parametrize("N", [2, 7, 12, 16])
def test_lane_per_column_kernel_explicit(B, N):
    M, K, bh, bw = 200, 333, 16, 64
    W = gen.dense_weight(M, K, seed=76)
    mask = gen.bcr_mask(M, K, bh, bw, compression=5, dist="uniform", seed=77)
    X = gen.normal_f32((K, N), 1.0, 78, 0)
    for variant in (0, 1, 2):  # default choice, values staged in registers, values streamed through shared memory
        check_spmm(B, W, mask, X, bh, bw, path=3, tile_n=variant)
        check_spmm(B, W, mask, X, bh, bw, bf16=True, path=3, tile_n=variant)


STREAM_CASES = [
    # M, K, bh, bw, generator kwargs: more bands than SMs, several bands per thread block, ragged edges
    (3000, 1500, 8, 32, dict(compression=4, dist="uniform")),
    (2500, 700, 16, 64, dict(compression=6, dist="zipf", empty_frac=0.1)),
    (20001, 96, 4, 16, dict(compression=3, dist="uniform")),   # > 32 bands per thread block: several batches
    (1190, 20000, 8, 32, dict(compression=16, dist="zipf")),   # vector too long for shared memory: gathered
]


@pytest.mark.parametrize("bf16", [False, True])
def test_small_n_edge_cases(B, bf16):
    """Default routing for N <= 16 on degenerate shapes: nothing kept at all, a single band shorter than a block, a
    matrix narrower than a block, one kept element, and the widest K the 16-bit column words can address."""
    for M, K, bh, bw, kw in [
        (40, 64, 8, 32, dict(compression=4, dist="uniform", empty_frac=1.0)),   # every block empty
        (5, 300, 8, 32, dict(compression=2, dist="uniform")),                   # one ragged band
        (100, 7, 4, 16, dict(compression=2, dist="uniform")),                   # K smaller than a block
        (64, 65536, 16, 64, dict(compression=64, dist="zipf")),                 # widest K of the chunk layout
    ]:
        W = gen.dense_weight(M, K, seed=180)
        mask = gen.bcr_mask(M, K, bh, bw, seed=181, **kw)
        for N in (1, 3, 16):
            X = gen.normal_f32((K, N), 1.0, 182, N)
            check_spmm(B, W, mask, X, bh, bw, bf16=bf16)
    W = gen.dense_weight(24, 96, seed=183)
    mask = np.zeros((24, 96), np.uint8)
    mask[9, 70] = 1  # a single kept element
    check_spmm(B, W, mask, gen.normal_f32((96, 1), 1.0, 184, 0), 8, 32, bf16=bf16)


@pytest.mark.parametrize("N", [1, 4, 9, 16])
@pytest.mark.parametrize("case", STREAM_CASES)
def test_streaming_kernel_explicit(B, case, N):
    M, K, bh, bw, kw = case
    W = gen.dense_weight(M, K, seed=170)
    mask = gen.bcr_mask(M, K, bh, bw, seed=171, **kw)
    mask[bh * 3:bh * 5] = 0  # two fully pruned bands
    X = gen.normal_f32((K, N), 1.0, 172, 0)
    check_spmm(B, W, mask, X, bh, bw, path=3, tile_n=2)
    check_spmm(B, W, mask, X, bh, bw, bf16=True, path=3, tile_n=2, y_bf16=(N == 4))


def test_spmm_strided_operands_and_errors(B):
    M, K, bh, bw, N = 64, 96, 8, 32, 20
    W = gen.dense_weight(M, K, seed=69)
    mask = gen.bcr_mask(M, K, bh, bw, compression=4, seed=70)
    h = B.grim_bcr_pack(W, mask, bh, bw, B.GRIM_F32, 0)
    Xfull = torch.randn(K, N + 7, device="cuda")
    Yfull = torch.zeros(M, N + 3, device="cuda")
    X, Y = Xfull[:, 2:2 + N], Yfull[:, 1:1 + N]  # ld > cols, unaligned start
    B.grim_bcr_spmm(h, X, Y)
    torch.cuda.synchronize()
    want = orc.spmm(W, mask, X.cpu().numpy())
    assert rel_fro(Y.cpu().numpy(), want) <= F32_TOL
    assert float(Yfull[:, 0].abs().max()) == 0.0 and float(Yfull[:, 1 + N:].abs().max()) == 0.0
    with pytest.raises(B.GrimError) as e:
        B.grim_bcr_spmm(h, torch.zeros(K + 1, N, device="cuda"), torch.zeros(M, N, device="cuda"))
    assert e.value.status == B.GRIM_ERR_SHAPE
    with pytest.raises(B.GrimError) as e:
        B.grim_bcr_spmm(h, torch.zeros(K, N, device="cuda", dtype=torch.bfloat16), torch.zeros(M, N, device="cuda"))
    assert e.value.status == B.GRIM_ERR_DTYPE
    with pytest.raises(B.GrimError) as e:
        B.grim_bcr_spmm(h, torch.zeros(K, N, device="cuda"), torch.zeros(M, N, device="cuda", dtype=torch.bfloat16))
    assert e.value.status == B.GRIM_ERR_DTYPE
    B.grim_bcr_destroy(h)


@pytest.mark.parametrize("case", [(4096, 1, 8.0, 8, 32, "uniform", False), (4096, 16, 16.0, 4, 16, "zipf", False),
                                  (2048, 128, 4.0, 16, 64, "zipf", True), (4096, 1, 4.0, 16, 64, "zipf", True),
                                  (1024, 1024, 8.0, 8, 32, "uniform", False)])
def test_sweep_points(B, case):
    M, N, c, bh, bw, dist, bf16 = case
    s = gen.sweep_case(M, N, c, bh, bw, dist, bf16=bf16)
    check_spmm(B, s["W"], s["mask"], s["X"], bh, bw, bf16=bf16, flags=1)


@pytest.mark.parametrize("N", [1, 4])
def test_streaming_kernel_chained_launches(B, N):
    """The streaming kernel is launched with programmatic stream serialization: a launch may begin (tables, barriers,
    first weight copies) while the launch before it still runs, and waits for it before it reads X or writes Y.  A chain
    of dependent products through two ping-pong buffers, queued without any host synchronisation, must therefore give
    what the oracle gives step by step - both the read-after-write (X of a step is Y of the step before) and the
    write-after-read (Y of a step is X of the step before) orders are exercised."""
    M = 2048
    s = gen.sweep_case(M, N, 4.0, 8, 32, "uniform")
    W = (s["W"] * 8.0).astype(np.float32)  # keeps the iterates at the same scale from step to step
    h = B.grim_bcr_pack(W, s["mask"], 8, 32, B.GRIM_F32, 1)
    try:
        bufs = [to_dev(s["X"]), torch.empty(M, N, device="cuda")]
        steps = 6
        for i in range(steps):
            B.grim_bcr_spmm_ex(h, bufs[i & 1], bufs[(i + 1) & 1], path=3, tile_n=2)
        torch.cuda.synchronize()
        assert B.grim_bcr_status(h) == B.GRIM_OK
        want = s["X"].astype(np.float64)
        for i in range(steps):
            want = orc.spmm(W, s["mask"], want.astype(np.float32)).astype(np.float64)
        got = bufs[steps & 1].cpu().numpy()
        assert rel_fro(got, want) <= 10 * F32_TOL, rel_fro(got, want)
    finally:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("reps", [3, -3])
def test_tune_returns_a_valid_choice(B, reps):
    """reps > 0 times back-to-back launches, reps < 0 launches after an L2 flush each (cold operands)."""
    s = gen.sweep_case(1024, 96, 8.0, 8, 32, "uniform")
    h = B.grim_bcr_pack(s["W"], s["mask"], 8, 32, B.GRIM_F32, 0)
    X = to_dev(s["X"])
    Y = torch.empty(1024, 96, device="cuda")
    best = B.grim_bcr_tune(h, X, Y, reps=reps)
    assert best["path"] in (1, 2, 3, 4) and best["ms"] > 0
    B.grim_bcr_spmm_ex(h, X, Y, tile_n=best["tile_n"], path=best["path"])
    torch.cuda.synchronize()
    assert rel_fro(Y.cpu().numpy(), orc.spmm(s["W"], s["mask"], s["X"])) <= F32_TOL
    # the answer is kept in the handle: the plain call now launches exactly what the explicit call launches
    Y.fill_(float("nan"))
    n0 = B.grim_launch_count()
    B.grim_bcr_spmm_ex(h, X, Y, tile_n=best["tile_n"], path=best["path"])
    n_explicit = B.grim_launch_count() - n0
    Y2 = torch.full_like(Y, float("nan"))
    B.grim_bcr_spmm(h, X, Y2)
    assert B.grim_launch_count() - n0 - n_explicit == n_explicit
    torch.cuda.synchronize()
    assert torch.equal(Y, Y2) or rel_fro(Y2.cpu().numpy(), Y.cpu().numpy()) <= 1e-6  # (a split multiply adds in any order)
    B.grim_bcr_destroy(h)


def test_regime_flags_keep_one_set_of_layouts(B):
    """A handle packed for narrow right-hand sides only multiplies N <= 16, one packed for wide ones N > 16; the other
    regime is refused before any launch, and each holds less device memory than a handle with every layout."""
    s = gen.sweep_case(1024, 64, 8.0, 8, 32, "uniform")
    X64, X4 = to_dev(s["X"]), to_dev(s["X"][:, :4])
    want = orc.spmm(s["W"], s["mask"], s["X"])
    free0 = torch.cuda.mem_get_info()[0]
    h_all = B.grim_bcr_pack(s["W"], s["mask"], 8, 32, B.GRIM_F32, 0)
    used_all = free0 - torch.cuda.mem_get_info()[0]
    B.grim_bcr_destroy(h_all)
    for flag, ok_x, bad_x in ((B.GRIM_PACK_NARROW_ONLY, X4, X64), (B.GRIM_PACK_WIDE_ONLY, X64, X4)):
        free1 = torch.cuda.mem_get_info()[0]
        h = B.grim_bcr_pack(s["W"], s["mask"], 8, 32, B.GRIM_F32, flag)
        assert free1 - torch.cuda.mem_get_info()[0] <= used_all
        Y = torch.full((1024, ok_x.shape[1]), float("nan"), device="cuda")
        B.grim_bcr_spmm(h, ok_x, Y)
        torch.cuda.synchronize()
        assert rel_fro(Y.cpu().numpy(), want[:, :ok_x.shape[1]]) <= F32_TOL
        with pytest.raises(B.GrimError) as e:
            B.grim_bcr_spmm(h, bad_x, torch.empty(1024, bad_x.shape[1], device="cuda"))
        assert e.value.status == B.GRIM_ERR_UNSUPPORTED
        B.grim_bcr_destroy(h)


# ---------------------------------------------------------------------------------------- convolution


def conv_col_norms(x, ksize, stride, pad):
    """||im2col column||_2 per output pixel: sqrt of the box-sum of x^2 over the receptive field."""
    xx = torch.from_numpy(np.asarray(x, np.float64) ** 2)
    ones = torch.ones(1, xx.shape[1], ksize, ksize, dtype=torch.float64)
    return torch.sqrt(torch.nn.functional.conv2d(xx, ones, stride=stride, padding=pad)).numpy()  # N,1,OH,OW


def check_conv(B, L, batch_x, *, ksize, stride, pad, bf16, relu=True, out_bf16=False, kernel_flags=0):
    W, mask, bias = L["W"], L["mask"], L["bias"]
    dt = B.GRIM_BF16 if bf16 else B.GRIM_F32
    x = gen.bf16_representable(batch_x) if bf16 else batch_x
    h = B.grim_bcr_pack(W, mask, L["bh"], L["bw"], dt, 0)
    try:
        xd = to_dev(x, bf16)
        Nb, C, H, Wd = x.shape
        OH = (H + 2 * pad - ksize) // stride + 1
        OW = (Wd + 2 * pad - ksize) // stride + 1
        out = torch.full((Nb, W.shape[0], OH, OW), float("nan"), device="cuda",
                         dtype=torch.bfloat16 if out_bf16 else torch.float32)
        if bf16:
            B.grim_bcr_reserve(h, Nb * OH * OW)
        B.grim_bcr_conv2d(h, xd, out, ksize, stride, pad, bias=to_dev(bias), relu=relu, kernel_flags=kernel_flags)
        torch.cuda.synchronize()
        assert B.grim_bcr_status(h) == B.GRIM_OK
        got = out.float().cpu().numpy().astype(np.float64)
        want = orc.conv2d(W, mask, x, bias, ksize=ksize, stride=stride, pad=pad, relu=relu, dtype=dt)
        Wm = orc.masked_weight(W, mask, dt)
        scale = np.linalg.norm(Wm, axis=1)[None, :, None, None] * conv_col_norms(x, ksize, stride, pad)
        assert_close(got, want, scale, bf16_in=bf16, out_bf16=out_bf16,
                     bias_abs=np.abs(bias.astype(np.float64))[None, :, None, None], what="conv")
        return got
    finally:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("geom", [(3, 1, 1), (3, 2, 1), (1, 1, 0), (5, 1, 2), (3, 1, 0)])
@pytest.mark.parametrize("bf16", [False, True])
def test_conv_small(B, geom, bf16):
    ks, stride, pad = geom
    L = gen.conv_layer(2, 12, 40, 13, ksize=ks, bh=8, bw=32, compression=4, seed=71)
    x = np.maximum(gen.normal_f32((3, 12, 13, 11), 1.0, 72, 0), 0)
    check_conv(B, L, x, ksize=ks, stride=stride, pad=pad, bf16=bf16)
    check_conv(B, L, x, ksize=ks, stride=stride, pad=pad, bf16=bf16, relu=False, out_bf16=bf16)


@pytest.mark.parametrize("bf16", [False, True])
def test_conv_11x11_and_1x1(B, bf16):
    """The large kernels of the paper's 3 x 3 against 11 x 11 comparison (Section 6.3), at stride 1 and at the stride 4
    of the classic first layer that uses them, and 1 x 1 kernels, which run as plain products per image (wide enough
    pixel counts to reach the tensor-core kernels with bf16)."""
    L = gen.conv_layer(2, 6, 48, 23, ksize=11, bh=8, bw=32, compression=5, seed=110)
    check_conv(B, L, L["x"], ksize=11, stride=1, pad=5, bf16=bf16)
    check_conv(B, L, L["x"], ksize=11, stride=4, pad=2, bf16=bf16, relu=False, out_bf16=bf16)
    L1 = gen.conv_layer(3, 96, 264, 24, ksize=1, bh=8, bw=32, compression=4, seed=111)
    check_conv(B, L1, L1["x"], ksize=1, stride=1, pad=0, bf16=bf16)
    check_conv(B, L1, L1["x"], ksize=1, stride=1, pad=0, bf16=bf16, relu=False, out_bf16=bf16)
    L2 = gen.conv_layer(2, 40, 72, 7, ksize=1, bh=4, bw=16, compression=3, seed=112)   # odd pixel count: unaligned rows
    check_conv(B, L2, L2["x"], ksize=1, stride=1, pad=0, bf16=bf16)


@pytest.mark.parametrize("bf16", [False, True])
def test_config3_conv_batch1(B, bf16):
    L = gen.conv_layer(1, 512, 512, 28, bf16=bf16)
    check_conv(B, L, L["x"], ksize=3, stride=1, pad=1, bf16=bf16)


def test_config3_conv_batch32_sampled(B):
    """Full-size launch (batch 32, the shape the benchmark times); the oracle checks 4 of the 32 images."""
    L = gen.conv_layer(32, 512, 512, 28)
    h = B.grim_bcr_pack(L["W"], L["mask"], 16, 64, B.GRIM_F32, 0)
    xd = to_dev(L["x"])
    out = torch.empty(32, 512, 28, 28, device="cuda")
    B.grim_bcr_conv2d(h, xd, out, 3, 1, 1, bias=to_dev(L["bias"]), relu=True)
    torch.cuda.synchronize()
    pick = [0, 7, 19, 31]
    want = orc.conv2d(L["W"], L["mask"], L["x"][pick], L["bias"], ksize=3, stride=1, pad=1, relu=True)
    assert rel_fro(out[pick].cpu().numpy(), want) <= F32_TOL
    B.grim_bcr_destroy(h)


def test_maxpool(B):
    x = torch.randn(2, 5, 8, 12, device="cuda")
    out = torch.empty(2, 5, 4, 6, device="cuda")
    B.grim_maxpool2x2(x, out)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().astype(np.float64), orc.maxpool2x2(x.cpu().numpy().astype(np.float64)))
    xb = x.to(torch.bfloat16)
    ob = torch.empty(2, 5, 4, 6, device="cuda", dtype=torch.bfloat16)
    B.grim_maxpool2x2(xb, ob)
    torch.cuda.synchronize()
    assert np.array_equal(ob.float().cpu().numpy().astype(np.float64),
                          orc.maxpool2x2(xb.float().cpu().numpy().astype(np.float64)))


def test_vgg_stack_small_image_per_layer(B):
    """Config-4 layer shapes at a 32x32 image: each layer is checked with the oracle fed the GPU's own
    previous-layer output (bf16 in, fp32 accumulate, bf16 out)."""
    net = gen.vgg16_stack(2, image=32)
    cur = to_dev(net["x"], True)
    for L in net["layers"]:
        h = B.grim_bcr_pack(L["W"], L["mask"], net["bh"], net["bw"], B.GRIM_BF16, 0)
        Nb, C, H, Wd = cur.shape
        out = torch.empty(Nb, L["cout"], H, Wd, device="cuda", dtype=torch.bfloat16)
        B.grim_bcr_conv2d(h, cur, out, 3, 1, 1, bias=to_dev(L["bias"]), relu=True)
        torch.cuda.synchronize()
        x_np = cur.float().cpu().numpy()
        want = orc.conv2d(L["W"], L["mask"], x_np, L["bias"], ksize=3, stride=1, pad=1, relu=True, dtype=orc.DTYPE_BF16)
        Wm = orc.masked_weight(L["W"], L["mask"], orc.DTYPE_BF16)
        scale = np.linalg.norm(Wm, axis=1)[None, :, None, None] * conv_col_norms(x_np, 3, 1, 1)
        assert_close(out.float().cpu().numpy(), want, scale, bf16_in=True, out_bf16=True,
                     bias_abs=np.abs(L["bias"].astype(np.float64))[None, :, None, None], what=f"vgg layer {L['cout']}")
        B.grim_bcr_destroy(h)
        if L["pool"]:
            pooled = torch.empty(Nb, L["cout"], H // 2, Wd // 2, device="cuda", dtype=torch.bfloat16)
            B.grim_maxpool2x2(out, pooled)
            cur = pooled
        else:
            cur = out


@pytest.mark.parametrize("layer", [0, 1, 4, 8, 12])
def test_vgg_full_size_layers(B, layer):
    """Config-4 layers at their real 224x224 sizes (batch 1, the launch shapes the benchmark times): first layer
    (K = 27, ragged), the widest pixel count, and one layer per resolution down to 14x14."""
    net = gen.vgg16_stack(1)
    L = net["layers"][layer]
    x = gen.bf16_representable(np.maximum(gen.normal_f32((1, L["cin"], L["hw"], L["hw"]), 1.0, 93, layer), 0))
    LL = dict(W=L["W"], mask=L["mask"], bias=L["bias"], bh=net["bh"], bw=net["bw"])
    check_conv(B, LL, x, ksize=3, stride=1, pad=1, bf16=True, out_bf16=True)


def test_conv_bf16_batch_crossing_images(B):
    """Tensor-core convolution with an image size that is not a multiple of the 8-pixel pieces or of the 256-column
    tile, several images, fp32 and bf16 outputs."""
    L = gen.conv_layer(5, 24, 72, 15, ksize=3, bh=8, bw=32, compression=5, seed=94)
    check_conv(B, L, L["x"], ksize=3, stride=1, pad=1, bf16=True)
    check_conv(B, L, L["x"], ksize=3, stride=1, pad=1, bf16=True, relu=False, out_bf16=True)


@pytest.mark.parametrize("shape", [(12, 12, 7), (8, 16, 9), (16, 10, 5), (24, 16, 3), (10, 14, 5), (14, 14, 3)])
@pytest.mark.parametrize("bh", [4, 8, 16])
def test_conv_bf16_staged_planes(B, shape, bh):
    """Tensor-core convolution on planes whose size is a multiple of 8 pixels, or of 4 (the variants that stage the
    input planes in shared memory by bulk copies / by 8-byte copies): 256-pixel tiles that meet two or three images, a
    ragged last tile, several K tiles, all block heights."""
    H, Wd, batch = shape
    C, Cout, bw = 20, 136, 32
    rng_seed = 300 + H + Wd + bh
    W = gen.dense_weight(Cout, C * 9, seed=rng_seed)
    mask = gen.bcr_mask(Cout, C * 9, bh, bw, compression=4, dist="uniform", seed=rng_seed + 1)
    bias = gen.normal_f32((Cout,), 0.1, rng_seed + 2, 0)
    x = np.maximum(gen.normal_f32((batch, C, H, Wd), 1.0, rng_seed + 3, 0), 0)
    L = dict(W=W, mask=mask, bias=bias, bh=bh, bw=bw)
    check_conv(B, L, x, ksize=3, stride=1, pad=1, bf16=True)
    check_conv(B, L, x, ksize=3, stride=1, pad=1, bf16=True, relu=False, out_bf16=True)


@pytest.mark.parametrize("shape", [(12, 12, 7), (8, 16, 9), (16, 10, 5), (24, 16, 3), (10, 14, 5), (14, 14, 3), (7, 9, 4), (15, 15, 5)])
@pytest.mark.parametrize("bh,cout", [(4, 136), (8, 300), (16, 520)])
def test_conv_bf16_paired_kernel(B, shape, bh, cout):
    """The paired tensor-core convolution asked for by name: planes staged by bulk copies (multiples of 8 pixels), by
    8-byte copies (multiples of 4) and read from global memory (others); tiles that meet two or three images, pixel
    counts that leave the odd block of a pair with a partial or an empty tile, one to five row tiles (odd counts give
    the last pair an empty partner), fp32 and bf16 outputs."""
    H, Wd, batch = shape
    C, bw = 20, 32
    rng_seed = 400 + H + Wd + bh
    W = gen.dense_weight(cout, C * 9, seed=rng_seed)
    mask = gen.bcr_mask(cout, C * 9, bh, bw, compression=4, dist="uniform", seed=rng_seed + 1)
    bias = gen.normal_f32((cout,), 0.1, rng_seed + 2, 0)
    x = np.maximum(gen.normal_f32((batch, C, H, Wd), 1.0, rng_seed + 3, 0), 0)
    L = dict(W=W, mask=mask, bias=bias, bh=bh, bw=bw)
    check_conv(B, L, x, ksize=3, stride=1, pad=1, bf16=True, kernel_flags=B.GRIM_CONV_PAIRED)
    check_conv(B, L, x, ksize=3, stride=1, pad=1, bf16=True, relu=False, out_bf16=True, kernel_flags=B.GRIM_CONV_PAIRED)


@pytest.mark.parametrize("y_bf16", [False, True])
def test_tensor_core_split_over_k(B, y_bf16):
    """Few output tiles and a long K: the tensor-core multiply is split over K (partial sums through the fp32
    scratch, second pass for the output), matrix and convolution forms, with pruned bands and a ragged last K tile."""
    M, K, bh, bw = 300, 3100, 8, 32
    W = gen.dense_weight(M, K, seed=310)
    mask = gen.bcr_mask(M, K, bh, bw, compression=6, dist="zipf", seed=311)
    mask[16:32] = 0
    X = gen.normal_f32((K, 304), 1.0, 312, 0)  # row stride a multiple of 16 bytes (TMA)
    check_spmm(B, W, mask, X, bh, bw, bf16=True, path=2, y_bf16=y_bf16)
    C, Cout = 176, 200
    Wc = gen.dense_weight(Cout, C * 9, seed=313)
    maskc = gen.bcr_mask(Cout, C * 9, 16, 64, compression=5, dist="uniform", seed=314)
    L = dict(W=Wc, mask=maskc, bias=gen.normal_f32((Cout,), 0.1, 315, 0), bh=16, bw=64)
    for H, Wd, batch in ((12, 12, 3), (7, 9, 2)):  # staged planes / planes read from global memory
        x = np.maximum(gen.normal_f32((batch, C, H, Wd), 1.0, 316, H), 0)
        check_conv(B, L, x, ksize=3, stride=1, pad=1, bf16=True, out_bf16=y_bf16)


# ---------------------------------------------------------------------------------------- GRU


def build_gru(B, m, max_T):
    hi, hh = [], []
    for lay in m["layers"]:
        hi.append(B.grim_bcr_pack(lay["W_ih"], lay["mask_ih"], m["bh"], m["bw"], B.GRIM_F32, 0))
        hh.append(B.grim_bcr_pack(lay["W_hh"], lay["mask_hh"], m["bh"], m["bw"], B.GRIM_F32, 0))
    g = B.grim_gru_create(hi, hh, [l["b_ih"] for l in m["layers"]], [l["b_hh"] for l in m["layers"]], max_T)
    return g, hi + hh


def check_gru(B, m, h0=None, grid_kernel=False):
    """Two passes on one handle against the oracle; returns the launches of the second."""
    T, H, L = m["T"], m["hidden"], len(m["layers"])
    g, handles = build_gru(B, m, T)
    try:
        if grid_kernel:  # a poll limit selects the cooperative-grid kernel instead of the cluster kernel
            B.grim_gru_debug_barrier(g, -1, 1 << 22)
        x = to_dev(m["x"])
        y = torch.full((T, H), float("nan"), device="cuda")
        hT = torch.full((L, H), float("nan"), device="cuda")
        for _ in range(2):  # the handle is reusable
            n0 = B.grim_launch_count()
            B.grim_gru_seq(g, x, y, h0=to_dev(h0) if h0 is not None else None, hT=hT)
            assert B.grim_gru_status(g) == B.GRIM_OK
            launches = B.grim_launch_count() - n0
        want_y, want_h = orc.gru_seq(m["layers"], m["x"], h0=h0)
        assert rel_fro(y.cpu().numpy(), want_y) <= F32_TOL, rel_fro(y.cpu().numpy(), want_y)
        assert rel_fro(hT.cpu().numpy(), want_h) <= F32_TOL
        return launches
    finally:
        B.grim_gru_destroy(g)
        for h in handles:
            B.grim_bcr_destroy(h)


@pytest.mark.parametrize("cfg", [(20, 64, 1, 7, 8, 32), (37, 128, 2, 13, 8, 32), (16, 96, 3, 5, 4, 16),
                                 (50, 256, 2, 9, 16, 64)])
def test_gru_small(B, cfg):
    in_f, H, L, T, bh, bw = cfg
    m = gen.gru_model(in_f, H, L, T, bh=bh, bw=bw, compression=4, seed=80)
    check_gru(B, m)
    h0 = gen.normal_f32((L, H), 0.5, 81, 0)
    check_gru(B, m, h0=h0)
    check_gru(B, m, h0=h0, grid_kernel=True)


def test_gru_four_layers_and_odd_hidden_size(B):
    """Four layers (run one after the other: the wavefront schedule is kept to three) against the oracle, and a
    hidden size that is a multiple of the block height but not of 4 is refused at creation."""
    check_gru(B, gen.gru_model(24, 128, 4, 70, bh=8, bw=32, compression=4, seed=97))
    m = gen.gru_model(12, 30, 1, 3, bh=6, bw=16, compression=2, seed=98)
    with pytest.raises(B.GrimError) as e:
        build_gru(B, m, 3)
    assert e.value.status == B.GRIM_ERR_UNSUPPORTED


@pytest.mark.parametrize("cfg", [(20, 592, 1, 9, 8, 32, 10), (16, 1024, 1, 6, 4, 16, 10), (16, 1024, 1, 6, 16, 64, 10), (16, 1024, 2, 70, 16, 64, 16),
                                 (30, 240, 2, 66, 16, 64, 8), (12, 272, 3, 67, 4, 16, 8), (9, 512, 1, 5, 4, 16, 8), (9, 1024, 1, 4, 8, 32, 8),
                                 (9, 1024, 1, 4, 16, 64, 8), (5, 20, 1, 3, 5, 16, 2), (7, 16, 2, 4, 16, 16, 2)])
def test_gru_block_shapes_and_hidden_sizes(B, cfg):
    """All block heights, unit groups that do not divide by the cluster, more columns per band than the register variants take."""
    in_f, H, L, T, bh, bw, rate = cfg
    check_gru(B, gen.gru_model(in_f, H, L, T, bh=bh, bw=bw, compression=rate, seed=201), h0=gen.normal_f32((L, H), 0.5, 202, 0))


def test_recurrent_kernel_tanh(B):
    """One step from a zero state on a zero input, update gate shut by its bias: the new state is tanh of the third gate's
    bias, element by element.  The kernel states 2.1 units in the last place against tanh itself; magnitudes from where tanh(x)
    is x to where it is 1, dense around the place where the two formulas meet."""
    H = 1024
    m = gen.gru_model(16, H, 1, 1, bh=8, bw=32, compression=10, seed=209)
    lay = m["layers"][0]
    ih, hh = (B.grim_bcr_pack(lay[w], lay[k], 8, 32, B.GRIM_F32, 0) for w, k in (("W_ih", "mask_ih"), ("W_hh", "mask_hh")))
    rng = np.random.default_rng(210)
    points = [np.geomspace(1e-30, 20.0, H), np.linspace(0.45, 0.55, H), np.linspace(0.0, 0.6, H), np.linspace(0.5, 10.0, H)]
    points += [rng.uniform(0.3, 3.0, H) for _ in range(4)]
    try:
        x, y = torch.zeros(1, 16, device="cuda"), torch.empty(1, H, device="cuda")
        worst = 0.0
        for v in points:
            v = (v * rng.choice([-1.0, 1.0], H)).astype(np.float32)
            b_ih = np.concatenate([np.zeros(H), np.full(H, -200.0), v]).astype(np.float32)
            g = B.grim_gru_create([ih], [hh], [b_ih], [np.zeros(3 * H, np.float32)], 1)
            B.grim_gru_seq(g, x, y)
            assert B.grim_gru_status(g) == B.GRIM_OK
            want = np.tanh(v.astype(np.float64))
            worst = max(worst, float(np.max(np.abs(y[0].cpu().numpy() - want) / np.spacing(np.abs(want).astype(np.float32)))))
            B.grim_gru_destroy(g)
        assert worst <= 2.1, worst
    finally:
        B.grim_bcr_destroy(ih)
        B.grim_bcr_destroy(hh)


@pytest.mark.parametrize("cfg", [(8, 136, 1, 60, 8, 32), (8, 528, 2, 90, 16, 64), (8, 592, 1, 60, 8, 32), (8, 260, 2, 100, 4, 16), (8, 392, 1, 61, 8, 32)])
def test_gru_unit_groups_for_fewer_blocks_than_the_largest_cluster(B, cfg):
    """17, 33, 74, 65 and 49 groups of units: dealt evenly to sixteen thread blocks they would leave seven, five, one, three
    and three of them without any.  Many steps, repeated: nothing times out and the results are right."""
    in_f, H, L, T, bh, bw = cfg
    m = gen.gru_model(in_f, H, L, T, bh=bh, bw=bw, compression=8, seed=206)
    for _ in range(3):
        check_gru(B, m, h0=gen.normal_f32((L, H), 0.5, 207, 0))


@pytest.mark.parametrize("cfg", [(9, 64, 2, 1, 8, 32, 4), (9, 64, 3, 2, 8, 32, 4), (12, 72, 2, 3, 4, 16, 3), (30, 1000, 2, 5, 8, 32, 10), (20, 1280, 3, 4, 16, 64, 30),
                                 (17, 1000, 2, 9, 4, 16, 16), (8, 16, 3, 150, 16, 16, 2)])
def test_gru_layers_in_one_launch(B, cfg):
    """Sequences shorter than what is brought ahead, more inputs to a projection than are in flight at once (1280), a last thread block
    with fewer units (1000); twice on each handle (the buffers between the layers start anew).  A transposing launch, the first layer's
    projection, the layers."""
    in_f, H, L, T, bh, bw, rate = cfg
    m = gen.gru_model(in_f, H, L, T, bh=bh, bw=bw, compression=rate, seed=441)
    assert check_gru(B, m) == 3
    assert check_gru(B, m, h0=gen.normal_f32((L, H), 0.5, 442, 0)) == 3


def test_gru_as_many_inputs_as_a_grid_has_rows(B):
    """2,097,120 inputs: the transposing launch has no rows of blocks left for filling the buffers between the layers."""
    in_f, H = 65535 * 32, 16
    m = gen.gru_model(64, H, 2, 3, bh=16, bw=64, compression=2, seed=481)
    lay, x = m["layers"][0], m["x"]
    at = np.concatenate([np.arange(32), np.arange(in_f - 32, in_f)])  # where the 64 inputs lie
    def wide(a):
        out = np.zeros((a.shape[0], in_f), a.dtype)
        out[:, at] = a
        return out
    big = dict(m, x=wide(x), layers=[dict(lay, W_ih=wide(lay["W_ih"]), mask_ih=wide(np.ones_like(lay["mask_ih"])))] + m["layers"][1:])
    g, handles = build_gru(B, big, 3)
    try:
        y = torch.full((3, H), float("nan"), device="cuda")
        B.grim_gru_seq(g, to_dev(big["x"]), y)
        assert B.grim_gru_status(g) == B.GRIM_OK
        want_y, _ = orc.gru_seq([dict(lay, mask_ih=np.ones_like(lay["mask_ih"]))] + m["layers"][1:], x)
        assert rel_fro(y.cpu().numpy(), want_y) <= F32_TOL
    finally:
        B.grim_gru_destroy(g)
        for h in handles:
            B.grim_bcr_destroy(h)


@pytest.mark.parametrize("cfg", [(30, 1040, 2, 5, 8, 32, 10), (20, 1536, 3, 4, 16, 64, 30), (17, 1200, 2, 9, 4, 16, 16)])
def test_gru_layers_beyond_the_registers(B, cfg):
    """Layers that no variant of the register-resident kernels holds: one after the other over the whole grid."""
    in_f, H, L, T, bh, bw, rate = cfg
    m = gen.gru_model(in_f, H, L, T, bh=bh, bw=bw, compression=rate, seed=441)
    assert check_gru(B, m) == 1 + 2 * L
    assert check_gru(B, m, h0=gen.normal_f32((L, H), 0.5, 442, 0)) == 1 + 2 * L


@pytest.mark.parametrize("cfg", [(40, 256, 2, 60, 8, 32, 8, 2), (20, 512, 3, 53, 8, 32, 10, 4), (20, 512, 2, 60, 8, 32, 16, 2)])
def test_gru_input_weights_denser_than_the_recurrent_ones(B, cfg):
    """The upper layers' W_ih would need a variant whose steps are much longer than W_hh's: the layers run chunk by chunk."""
    in_f, H, L, T, bh, bw, rate, rate_ih = cfg
    m = gen.gru_model(in_f, H, L, T, bh=bh, bw=bw, compression=rate, seed=461)
    for l, lay in enumerate(m["layers"][1:]):
        lay["mask_ih"] = gen.bcr_mask(3 * H, H, bh, bw, compression=rate_ih, seed=462 + l)
    pieces = 2
    assert check_gru(B, m, h0=gen.normal_f32((L, H), 0.5, 463, 0)) == 2 + (2 * L - 1) * pieces


@pytest.mark.parametrize("cfg", [(37, 128, 2, 33, 4, 16), (20, 96, 1, 31, 16, 32), (64, 160, 3, 64, 16, 64), (9, 60, 2, 2, 5, 16), (500, 64, 2, 7, 8, 32)])
def test_gru_batched_step_block_shapes(B, cfg):
    """Batches around a tile of 32 sequences, block heights, inputs wider and narrower than the state."""
    in_f, H, L, batch, bh, bw = cfg
    m = gen.gru_model(in_f, H, L, 2, bh=bh, bw=bw, compression=3, seed=203)
    g, handles = build_gru(B, m, 2 * batch)
    try:
        x, h0 = gen.normal_f32((batch, in_f), 1.0, 204, 0), gen.normal_f32((L, batch, H), 0.5, 205, 0)
        h, y = to_dev(h0), torch.empty(batch, H, device="cuda")
        B.grim_gru_step(g, to_dev(x), h, y)
        assert B.grim_gru_status(g) == B.GRIM_OK
        for b in range(batch):
            yb, hb = orc.gru_seq(m["layers"], x[b:b + 1], h0=h0[:, b])
            assert rel_fro(y[b].cpu().numpy(), yb[0]) <= F32_TOL and rel_fro(h[:, b].cpu().numpy(), hb) <= F32_TOL
    finally:
        B.grim_gru_destroy(g)
        for hd in handles:
            B.grim_bcr_destroy(hd)


@pytest.mark.parametrize("grid_kernel", [False, True])
def test_config2_gru_full(B, grid_kernel):
    check_gru(B, gen.gru_model(), grid_kernel=grid_kernel)


@pytest.mark.parametrize("chunks", [1, 2, 5, 8])
def test_gru_layer_pipelining_gives_the_same_result(B, chunks):
    """Three layers cut into `chunks` pieces in time and run as a wavefront on internal streams: same outputs and
    final states as the oracle, with and without an initial state, on a sequence length that does not divide.  A transposing
    launch, the first layer's projection, and per piece a recurrent launch per layer and a projection per upper one
    (pieces are multiples of four steps: eight of 53 are seven)."""
    m = gen.gru_model(30, 128, 3, 53, bh=8, bw=32, compression=4, seed=95)
    T, H, L = m["T"], m["hidden"], 3
    g, handles = build_gru(B, m, T)
    try:
        B.grim_gru_set_pipeline(g, chunks)
        h0 = gen.normal_f32((L, H), 0.5, 96, 0)
        for init in (None, h0):
            y = torch.full((T, H), float("nan"), device="cuda")
            hT = torch.full((L, H), float("nan"), device="cuda")
            n0 = B.grim_launch_count()
            B.grim_gru_seq(g, to_dev(m["x"]), y, h0=to_dev(init) if init is not None else None, hT=hT)
            assert B.grim_launch_count() - n0 == 2 + 5 * min(chunks, 7)
            assert B.grim_gru_status(g) == B.GRIM_OK
            want_y, want_h = orc.gru_seq(m["layers"], m["x"], h0=init)
            assert rel_fro(y.cpu().numpy(), want_y) <= F32_TOL
            assert rel_fro(hT.cpu().numpy(), want_h) <= F32_TOL
    finally:
        B.grim_gru_destroy(g)
        for h in handles:
            B.grim_bcr_destroy(h)


@pytest.mark.parametrize("cfg", [(153, 1024, 2, 32), (37, 128, 3, 5), (20, 64, 1, 1)])
def test_gru_batched_step(B, cfg):
    """One time step for a batch of sequences (the paper's timed GRU shape is sequence length 1, batch 32), two steps in a
    row so that the carried state is used: against the oracle run per batch element."""
    in_f, H, L, batch = cfg
    m = gen.gru_model(in_f, H, L, 2, compression=10 if H == 1024 else 4, seed=99)
    g, handles = build_gru(B, m, 2 * batch + 2)
    try:
        xs = [gen.normal_f32((batch, in_f), 1.0, 100, t) for t in range(2)]
        h = to_dev(gen.normal_f32((L, batch, H), 0.5, 101, 0))
        h_np = h.cpu().numpy().astype(np.float64)
        y = torch.full((batch, H), float("nan"), device="cuda")
        for t in range(2):
            B.grim_gru_step(g, to_dev(xs[t]), h, y)
            torch.cuda.synchronize()
            want_y = np.empty((batch, H))
            for b in range(batch):
                yb, hb = orc.gru_seq(m["layers"], xs[t][b:b + 1], h0=h_np[:, b])
                want_y[b], h_np[:, b] = yb[0], hb
            assert rel_fro(y.cpu().numpy(), want_y) <= F32_TOL
            assert rel_fro(h.cpu().numpy(), h_np) <= F32_TOL
        with pytest.raises(B.GrimError) as e:
            B.grim_gru_step(g, torch.zeros(2 * batch + 2, in_f, device="cuda"), torch.zeros(L, 2 * batch + 2, H, device="cuda"))
        assert e.value.status == B.GRIM_ERR_SHAPE
    finally:
        B.grim_gru_destroy(g)
        for hd in handles:
            B.grim_bcr_destroy(hd)


def test_gru_bounded_wait_reports_timeout(B):
    """One thread block stays away from the step barrier: every wait runs out after a small bound, the
    kernel returns by itself and the status word says so; afterwards the handle works normally."""
    m = gen.gru_model(20, 256, 1, 6, bh=8, bw=32, compression=4, seed=82)
    g, handles = build_gru(B, m, 6)
    x = to_dev(m["x"])
    y = torch.zeros(6, 256, device="cuda")
    B.grim_gru_debug_barrier(g, 1, 20000)
    B.grim_gru_seq(g, x, y)
    assert B.grim_gru_status(g) == B.GRIM_ERR_TIMEOUT
    B.grim_gru_debug_barrier(g, -1, 0)
    B.grim_gru_seq(g, x, y)
    assert B.grim_gru_status(g) == B.GRIM_OK
    want_y, _ = orc.gru_seq(m["layers"], m["x"])
    assert rel_fro(y.cpu().numpy(), want_y) <= F32_TOL
    B.grim_gru_destroy(g)
    for h in handles:
        B.grim_bcr_destroy(h)


@pytest.mark.parametrize("L,T", [(2, 1), (2, 7), (3, 12)])
def test_gru_bounded_waits_between_layers_report_timeout(B, L, T):
    """What the upper layers of a single launch wait for never comes: their waits run out, the launch ends and the status word says
    so; afterwards the handle works normally."""
    m = gen.gru_model(20, 256, L, T, bh=8, bw=32, compression=4, seed=83)
    g, handles = build_gru(B, m, T)
    x = to_dev(m["x"])
    y = torch.zeros(T, 256, device="cuda")
    B.grim_gru_debug_barrier(g, -2, 2000)
    B.grim_gru_seq(g, x, y)
    assert B.grim_gru_status(g) == B.GRIM_ERR_TIMEOUT
    B.grim_gru_debug_barrier(g, -1, 0)
    B.grim_gru_seq(g, x, y)
    assert B.grim_gru_status(g) == B.GRIM_OK
    want_y, _ = orc.gru_seq(m["layers"], m["x"])
    assert rel_fro(y.cpu().numpy(), want_y) <= F32_TOL
    B.grim_gru_destroy(g)
    for h in handles:
        B.grim_bcr_destroy(h)
