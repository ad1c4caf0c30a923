"""GPU parity of the GEMM kernel for few activation rows (every warp alone on a slice of K) against the FP64 oracle, at the sizes
where its division can go wrong: one to eight rows, up to 16, 32 and several blocks of rows; units of 16 and 32 columns that end
within the matrix; slices that end within 64 k, blocks of a cluster with fewer k than the others, more lanes than units; both
layouts of both operands with padded leading dimensions, accumulation, one scale per column; the longest K.  And the forms of the
kernel that decodes the weights for small products and for the last round of tiles, and the expansion of many activations.

Which kernel runs is asked for (hif8_gemm_path_policy) and seen by the number of launches.

Tolerance per output: 1e-5 * S of the method's statement, one FP32 rounding of the sum, and half a unit in the last place of BF16.
"""
import numpy as np
import pytest
import torch

import paper_2409_16626_b200 as H
import workloads as W
from oracle import hif8_oracle as O

from gpu_util import bf16_half_ulp, gemm_path, to_dev

pytestmark = pytest.mark.gpu


def codes(shape, seed):
    t = W.random_codes(shape, seed=seed)
    t[(t == 0x80) | ((t & 0x7F) == 0x6F)] = 0x33
    return t


def padded(t, extra, multiple=16):
    out = np.full((t.shape[0], (t.shape[1] + multiple - 1) // multiple * multiple + extra), 0x7B, dtype=np.uint8)
    out[:, :t.shape[1]] = t
    return out


@pytest.mark.parametrize("c_dtype,accumulate,channel", [(H.F32, 0, 0), (H.BF16, 0, 1), (H.F32, 1, 1), (H.BF16, 1, 0)])
@pytest.mark.parametrize("w_is_nk", [0, 1])
@pytest.mark.parametrize("a_is_km", [0, 1])
@pytest.mark.parametrize("shape", [(1, 16, 16), (8, 44, 80), (9, 512, 512), (16, 1004, 272), (17, 40, 2064), (32, 328, 1040), (33, 516, 64), (100, 96, 144),
                                   (4, 48, "longest"), (16, 256, 8192), (13, 7168, 256), (24, 1004, 4112), (130, 2000, 528), (260, 1004, 1040)])
def test_gemm_few_rows(shape, a_is_km, w_is_nk, c_dtype, accumulate, channel):
    # (the last three: several units of columns a warp one after the other, up to 32 rows a block in every layout, clusters)
    M, N, K = shape
    if K == "longest":  # 128 warps of a cluster with one to four blocks of 64 k each; a block more has no room
        K = 8192 * ((4 if w_is_nk else 2) // (2 if a_is_km else 1))
    Amk, Wkn = codes((M, K), M + K), codes((K, N), N + K + 1)
    A = padded(np.ascontiguousarray(Amk.T) if a_is_km else Amk, 16)
    Wq = padded(np.ascontiguousarray(Wkn.T) if w_is_nk else Wkn, 16)
    rng = np.random.default_rng(M)
    ldc = (N + 7) // 8 * 8 + 8
    c0 = torch.from_numpy((rng.standard_normal((M, ldc)) * 50).astype(np.float32)).cuda()
    C = c0.clone() if c_dtype == H.F32 else c0.bfloat16()
    c0 = C.float().cpu().numpy().astype(np.float64)
    sw = rng.integers(-9, 9, N).astype(np.int32) if channel else -4
    ws = torch.full((256,), 0xFF, dtype=torch.uint8, device="cuda")
    before = H.hif8_launch_count()
    with gemm_path(H.GEMM_PATH_WARP):
        H.hif8_gemm_ex(to_dev(A), A.shape[1], a_is_km, to_dev(Wq), Wq.shape[1], w_is_nk, C, ldc, c_dtype, M, N, K, torch.tensor([3], dtype=torch.int32, device="cuda"),
                       None if channel else torch.tensor([sw], dtype=torch.int32, device="cuda"), to_dev(sw.view(np.uint32)) if channel else None, accumulate, ws, 256)
    assert H.hif8_gemm_status(ws) == 0 and H.hif8_launch_count() == before + 1
    out = C.float().cpu().numpy().astype(np.float64)
    assert np.array_equal(out[:, N:], c0[:, N:])             # padding columns untouched
    n = min(M * N, 40000)                                     # every output, or the last columns of every row and a sample
    rows, cols = np.divmod(np.arange(M * N), N) if n == M * N else (np.concatenate([rng.integers(0, M, n), np.repeat(np.arange(M), 64)]),
                                                                    np.concatenate([rng.integers(0, N, n), np.tile(np.arange(N - 64, N), M)]))
    P, S = O.gemm_entries_ex(Amk, 0, Wkn, 0, 3, sw, rows, cols)
    want = P + c0[rows, cols] if accumulate else P
    tol = 1e-5 * S + 2.0 ** -24 * np.abs(want)
    if c_dtype == H.BF16:
        tol = tol + bf16_half_ulp(np.abs(want) + tol)
    assert np.all(np.abs(out[rows, cols] - want) <= tol)


def test_gemm_few_rows_is_refused_where_it_has_no_division():
    # the setting that asks for this kernel; by itself the library takes another one for these products
    buf, ws = torch.zeros(1 << 22, dtype=torch.uint8, device="cuda"), torch.empty(256, dtype=torch.uint8, device="cuda")
    C = torch.zeros(1 << 20, dtype=torch.float32, device="cuda")
    for km, nk, M, N, K in ((0, 0, 4, 48, 16400), (0, 1, 4, 48, 32784), (1, 0, 4, 48, 8208), (1, 1, 4, 48, 16400), (0, 0, 4, 42, 64), (0, 0, 33, 48, 8208)):
        call = lambda: H.hif8_gemm_ex(buf, 16 if km else K, km, buf, K if nk else 48, nk, C, 48, H.F32, M, N, K, None, None, None, 0, ws, 256, check=False)
        with gemm_path(H.GEMM_PATH_WARP):
            if (M, nk, km) == (33, 0, 0):
                assert call() == 0  # (16 rows a block reach twice as far as 32)
            else:
                assert call() == 6  # HIF8_ERR_SHAPE
        assert call() == 0 and H.hif8_gemm_status(ws) == 0


@pytest.mark.parametrize("shape", [(1, 512, 512), (16, 2048, 2048), (128, 512, 1024)])
def test_gemm_few_rows_is_taken_by_itself(shape):
    # with room for both operands every other kernel takes two launches or more here
    M, N, K = shape
    A, W = torch.full((M * K,), 0x08, dtype=torch.uint8, device="cuda"), torch.full((N * K,), 0x08, dtype=torch.uint8, device="cuda")
    C, wsb = torch.zeros(M, N, dtype=torch.float32, device="cuda"), H.hif8_workspace_bytes(H.WS_GEMM, M * K + K * N)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    before = H.hif8_launch_count()
    H.hif8_gemm(A, K, W, K, 1, C, N, H.F32, M, N, K, None, None, ws, wsb)
    assert H.hif8_launch_count() == before + 1 and bool((C == K).all())
    with gemm_path(H.GEMM_PATH_EXPAND_A):
        H.hif8_gemm(A, K, W, K, 1, C, N, H.F32, M, N, K, None, None, ws, wsb)
    assert H.hif8_launch_count() >= before + 3 and bool((C == K).all())


@pytest.mark.parametrize("w_is_nk", [0, 1])
def test_gemm_few_rows_specials_and_repeats(w_is_nk):
    # NaN and Inf reach their row and column and nothing else, and the order of the sums does not depend on which warp is first
    M, N, K = 16, 520, 1040
    A, Wkn = codes((M, K), 1), codes((K, N), 2)
    A[3, 5], A[7, 1039], Wkn[1030, 517] = 0x80, 0x6F, 0x80
    Wkn[1039] = 0x08
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    Wq = np.ascontiguousarray(Wkn.T) if w_is_nk else padded(Wkn, 0)
    outs = []
    for _ in range(4):
        C = torch.zeros(M, N, dtype=torch.float32, device="cuda")
        with gemm_path(H.GEMM_PATH_WARP):
            H.hif8_gemm(to_dev(A), K, to_dev(Wq), Wq.shape[1], w_is_nk, C, N, H.F32, M, N, K, None, None, ws, 256)
        assert H.hif8_gemm_status(ws) == 0
        outs.append(C.cpu().numpy())
    out = outs[0]
    assert all(np.array_equal(out, o, equal_nan=True) for o in outs)
    nan = np.zeros((M, N), bool)
    nan[3], nan[:, 517] = True, True
    assert np.array_equal(np.isnan(out), nan)
    rest = np.delete(np.arange(N), 517)
    assert np.all(np.isposinf(out[7][rest]))
    assert np.all(np.isfinite(np.delete(out, [3, 7], axis=0)[:, rest]))


@pytest.mark.parametrize("shape,form", [((65, 512, 2048), "rows"), ((250, 2064, 1040), "rows"), ((250, 2064, 1040), "columns"), ((1024, 528, 528), "rows"),
                                        ((1024, 528, 528), "columns")])
def test_gemm_pieces_of_activation_rows(shape, form):
    # products of few tiles: the weights kernel in smaller pieces of activation rows than one of 256, activations as bytes
    M, N, K = shape
    M = M if form == "rows" else (M + 15) // 16 * 16
    Amk, Wkn = codes((M, K), M), codes((K, N), N)
    A = Amk if form == "rows" else np.ascontiguousarray(Amk.T)
    C = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    wsb = H.hif8_workspace_bytes(H.WS_GEMM, M * K + K * N)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    before = H.hif8_launch_count()
    with gemm_path(H.GEMM_PATH_NO_WARP):
        H.hif8_gemm_ex(to_dev(A), A.shape[1], form == "columns", to_dev(Wkn), N, 0, C, N, H.F32, M, N, K, None, None, None, 0, ws, wsb)
    assert H.hif8_gemm_status(ws) == 0 and H.hif8_launch_count() == before + 1
    rng = np.random.default_rng(3)
    rows, cols = np.concatenate([rng.integers(0, M, 30000), np.repeat(np.arange(M), 16)]), np.concatenate([rng.integers(0, N, 30000), np.tile(np.arange(N - 16, N), M)])
    P, S = O.gemm_entries(Amk, Wkn, False, 0, 0, rows, cols)
    assert np.all(np.abs(C.cpu().numpy().astype(np.float64)[rows, cols] - P) <= 1e-5 * S)


@pytest.mark.parametrize("accumulate", [0, 1])
@pytest.mark.parametrize("shape,form", [((1216, 3904, 1040), "rows"), ((1216, 3904, 1040), "columns"), ((304, 10000, 1552), "expanded"), ((2400, 4096, 1040), "rows")] +
                         [(s, f) for s in ((1200, 3904, 1552), (512, 10000, 1552), (2400, 4096, 2064)) for f in ("rows", "columns", "expanded")])
def test_gemm_last_round_in_parts(shape, form, accumulate):
    # 80 to 160 tiles of up to 256 activation rows on 74 pairs: the last ones in parts of fewer rows, some split along K, in a
    # launch of their own; the last part of a tile and the last piece of the matrix shorter than the others; more pieces than one
    # group of eight.  Each output is written (or added to) once.
    M, N, K = shape
    Amk, Wkn = codes((M, K), M), codes((K, N), N)
    A = np.ascontiguousarray(Amk.T) if form == "columns" else Amk
    rng = np.random.default_rng(M)
    c0 = (rng.standard_normal((M, N)) * 50).astype(np.float32)
    C = torch.from_numpy(c0.copy()).cuda()
    wsb = 256 + (2 * M * K + 255) // 256 * 256 if form == "expanded" else 256
    ws = torch.full((wsb,), 0xFF, dtype=torch.uint8, device="cuda")
    before = H.hif8_launch_count()
    with gemm_path(H.GEMM_PATH_EXPAND_A):
        H.hif8_gemm_ex(to_dev(A), A.shape[1], form == "columns", to_dev(Wkn), N, 0, C, N, H.F32, M, N, K, torch.tensor([3], dtype=torch.int32, device="cuda"),
                       torch.tensor([-4], dtype=torch.int32, device="cuda"), None, accumulate, ws, wsb)
    assert H.hif8_gemm_status(ws) == 0
    assert H.hif8_launch_count() == before + (3 if form == "expanded" else 2)
    rows = np.concatenate([rng.integers(0, M, 40000), np.repeat(np.arange(M), 24)])
    cols = np.concatenate([rng.integers(0, N, 40000), np.tile(np.arange(N - 24, N), M)])
    P, S = O.gemm_entries(Amk, Wkn, False, 3, -4, rows, cols)
    want = P + c0[rows, cols] if accumulate else P
    assert np.all(np.abs(C.cpu().numpy().astype(np.float64)[rows, cols] - want) <= 1e-5 * S + 2.0 ** -24 * np.abs(want))


@pytest.mark.parametrize("shape", [(1029, 272, 4112), (1024, 272, 4096), (4001, 144, 1056)])
def test_gemm_many_activations_expanded(shape):
    # four million activations and more: the expansion with a table per lane, in blocks of 16384; lengths that end within a block
    # and at the end of one
    M, N, K = shape
    assert M * K >= 1 << 22
    Amk, Wkn = codes((M, K), M), codes((K, N), N)
    wsb = 256 + (2 * M * K + 255) // 256 * 256
    ws = torch.full((wsb,), 0xFF, dtype=torch.uint8, device="cuda")
    C = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    with gemm_path(H.GEMM_PATH_EXPAND_A):
        H.hif8_gemm(to_dev(Amk), K, to_dev(Wkn), N, 0, C, N, H.F32, M, N, K, None, None, ws, wsb)
    assert H.hif8_gemm_status(ws) == 0
    table = torch.from_numpy(O.decode(np.arange(256, dtype=np.uint8), H.BF16, 0).view(np.int16)).cuda()
    assert torch.equal(ws[256:256 + 2 * M * K].view(torch.int16), table[to_dev(Amk).view(-1).long()])  # every activation, bit for bit
    rng = np.random.default_rng(3)
    rows, cols = np.concatenate([rng.integers(0, M, 20000), np.repeat(np.arange(M), 4)]), np.concatenate([rng.integers(0, N, 20000), np.tile(np.arange(N - 4, N), M)])
    P, S = O.gemm_entries(Amk, Wkn, False, 0, 0, rows, cols)
    assert np.all(np.abs(C.cpu().numpy().astype(np.float64)[rows, cols] - P) <= 1e-5 * S)
