"""GPU parity of how the single-layer kernel moves 8-bit rows, against the CPU oracle, bit-exact.  By the epilogue: pitches,
offsets and pointers on the 16-byte grid but off the 32-byte one, odd numbers of 16-column chunks, residual rows of another
alignment than the output's, one tile and several per CTA, CTA pairs.  Through tile buffers (long launches with wide tiles and
short reductions): every operand path, one and two buffers a group, ragged tiles of rows and of columns, channel
slices, with and without a residual; residuals of fp32 outputs.  Bytes beside the rows stay as they are."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8, F32 = 0, 1, 3

CASES = [
    # name, N,H,W,C,K,R,pad, y type, residual, pitch - K, channel offset, output shift, residual shift (bytes)
    ("k16", 2, 20, 21, 64, 16, 3, 1, U8, True, 0, 0, 0, 0),
    ("k48_odd_chunks", 3, 45, 45, 64, 48, 1, 0, U8, True, 0, 0, 0, 0),
    ("k64_slice_16", 4, 33, 33, 64, 64, 1, 0, U8, True, 32, 16, 0, 0),
    ("k64_pitch_80", 4, 60, 60, 64, 64, 3, 1, S8, True, 16, 0, 0, 0),
    ("k96_output_off", 2, 30, 31, 96, 96, 3, 1, U8, True, 0, 0, 16, 0),
    ("k96_residual_off", 2, 30, 31, 96, 96, 3, 1, U8, True, 0, 0, 0, 16),
    ("k112_short", 1, 14, 14, 320, 112, 1, 0, U8, True, 16, 0, 0, 0),
    ("k208_long_buffered", 16, 57, 57, 64, 208, 1, 0, S8, True, 0, 0, 0, 0),
    ("k256_one_tile_a_cta", 8, 28, 28, 256, 256, 3, 1, U8, True, 0, 0, 0, 0),
    ("k48_long", 40, 45, 45, 64, 48, 1, 0, S8, True, 16, 16, 16, 0),
    ("k160_pairs", 32, 44, 44, 128, 160, 3, 1, U8, True, 16, 16, 0, 0),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_rows_in_global_memory_match_oracle(q8, case):
    name, N, H, W, C, K, R, pad, ytype, res, extra, c_off, yshift, rshift = case
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, R, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, (1, 1), (pad, pad), (1, 1), threads=8)
    resid = g.integers(0, 256, acc.shape, dtype=np.uint8)
    scale = np.float32(100.0 / max(1, np.abs(acc).max()))
    want = o.epilogue(acc, scale, resid, 0.37, ytype == U8, o.U8 if ytype == U8 else o.S8)
    ldc = K + extra
    d = q8.make_conv_desc(N, H, W, C, K, R, R, (1, 1), (pad, pad), (1, 1), U8, U8, ytype, ytype == U8, 1, ldc, c_off)
    plan = q8.q8_conv2d_query_plan(d, res)
    assert plan.kernel == q8.Q8_KERNEL_TMA and not plan.moved_rows and plan.cta_pair == ("pairs" in name)
    assert (q8.q8_conv2d_query_row_buffers(d, None, res) > 0) == ("buffered" in name)
    rows = N * H * W
    buf = torch.full((64 + rows * ldc + 64,), 7, dtype=q8.TORCH_DTYPES[ytype], device="cuda")
    y = buf[32 + yshift:32 + yshift + rows * ldc].view(N, H, W, ldc)
    rbuf = torch.zeros(rows * K + 32, dtype=torch.uint8, device="cuda")
    rd = rbuf[rshift:rshift + rows * K].view(N, H, W, K)
    rd.copy_(torch.from_numpy(resid).cuda())
    q8.q8_conv2d(d, torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), torch.from_numpy(bias).cuda(),
                 torch.tensor([scale], device="cuda"), rd, 0.37, y)
    q8.q8_read_status()
    got = y.cpu().numpy()
    assert np.array_equal(got[..., c_off:c_off + K], want)
    assert (got[..., :c_off] == 7).all() and (got[..., c_off + K:] == 7).all()
    assert (buf[:32 + yshift] == 7).all() and (buf[32 + yshift + rows * ldc:] == 7).all()


BUFFERED = [
    # name, N,H,W,C,K,R,stride,pad, y type, residual, per channel, pitch - K, channel offset, tile width, CTA pair, buffers
    ("matrix_no_residual", 47, 57, 57, 64, 256, 1, 1, 0, S8, None, False, 0, 0, 128, 0, 8),
    ("matrix_slice_s8_residual", 12, 57, 57, 64, 256, 1, 1, 0, S8, "s8", True, 48, 16, 128, 0, 8),
    ("matrix_one_a_group", 12, 57, 57, 256, 256, 1, 1, 0, U8, "u8", False, 0, 0, 128, 0, 4),
    ("ragged_columns_208", 25, 57, 57, 32, 208, 1, 1, 0, U8, "u8", True, 16, 0, 112, 0, 8),
    ("ragged_columns_272", 12, 57, 57, 64, 272, 1, 1, 0, S8, "u8", False, 0, 0, 96, 0, 8),
    ("halo_64_columns", 64, 56, 56, 16, 64, 3, 1, 1, U8, None, True, 0, 0, 64, 0, 8),
    ("halo_ragged_edges", 22, 37, 41, 32, 192, 3, 1, 1, U8, "u8", False, 64, 32, 96, 0, 8),
    ("halo_one_a_group", 12, 57, 57, 32, 256, 3, 1, 1, S8, "u8", True, 0, 0, 128, 0, 4),
    ("halo_streamed_weights", 47, 37, 41, 64, 160, 3, 1, 1, U8, "u8", False, 0, 0, 80, 0, 4),
    ("im2col", 30, 75, 75, 32, 256, 3, 2, 0, U8, "s8", False, 0, 0, 128, 0, 4),
    ("pairs_odd_tiles", 23, 37, 41, 64, 256, 3, 1, 1, U8, "u8", True, 16, 16, 128, 1, 4),
    ("pairs_no_residual", 70, 37, 41, 64, 256, 3, 1, 1, S8, None, False, 0, 0, 128, 1, 4),
    ("matrix_f32", 12, 57, 57, 64, 256, 1, 1, 0, F32, "u8", False, 8, 4, 128, 0, 8),
    ("matrix_f32_two_tiles", 4, 57, 57, 64, 256, 1, 1, 0, F32, "s8", True, 0, 0, 128, 0, 8),
    ("matrix_f32_64_columns", 60, 57, 57, 32, 64, 1, 1, 0, F32, "u8", True, 0, 0, 64, 0, 8),
    ("halo_f32_ragged_edges", 22, 37, 41, 32, 192, 3, 1, 1, F32, "s8", True, 4, 0, 96, 0, 8),
    ("halo_f32_256_columns", 25, 28, 28, 128, 256, 3, 1, 1, F32, "u8", False, 0, 0, 256, 0, 2),
    ("pairs_shared_groups", 47, 37, 41, 128, 160, 3, 1, 1, S8, "s8", False, 0, 0, 160, 1, 2),
]


@pytest.mark.parametrize("case", BUFFERED, ids=[c[0] for c in BUFFERED])
def test_rows_through_tile_buffers_match_oracle(q8, case):
    name, N, H, W, C, K, R, st, pad, ytype, res, per_channel, extra, c_off, tile_n, pair, buffers = case
    ldc, res_type = K + extra, S8 if res == "s8" else U8
    d = q8.make_conv_desc(N, H, W, C, K, R, R, (st, st), (pad, pad), (1, 1), U8, res_type, ytype, ytype == U8, K if per_channel else 1,
                          ldc, c_off)
    plan = q8.q8_conv2d_query_plan(d, res is not None)
    assert (plan.kernel, plan.tile_n, plan.cta_pair) == (q8.Q8_KERNEL_TMA, tile_n, pair)
    assert q8.q8_conv2d_query_row_buffers(d, None, res is not None) == buffers
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, R, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, (st, st), (pad, pad), (1, 1), threads=8)
    resid = None if res is None else g.integers(0, 256, acc.shape, dtype=np.uint8).view(np.int8 if res == "s8" else np.uint8)
    scale = (g.uniform(0.5, 1.5, K if per_channel else 1) * 100.0 / max(1, np.abs(acc).max())).astype(np.float32)
    want = o.epilogue(acc, scale if per_channel else scale[0], resid, 0.37, ytype == U8, {U8: o.U8, S8: o.S8, F32: o.F32}[ytype])
    args = [torch.from_numpy(a).cuda() for a in (x, w, bias, scale)]
    rd = None if resid is None else torch.from_numpy(resid).cuda()
    y = torch.full((*acc.shape[:3], ldc), 7, dtype=q8.TORCH_DTYPES[ytype], device="cuda")
    for _ in range(2):   # twice: the second launch follows the first in the stream
        q8.q8_conv2d(d, *args, rd, 0.37 if res else 0.0, y)
    q8.q8_read_status()
    got = y.cpu().numpy()
    assert np.ascontiguousarray(got[..., c_off:c_off + K]).tobytes() == want.tobytes()
    assert (got[..., :c_off] == 7).all() and (got[..., c_off + K:] == 7).all()
