"""GPU parity of the epilogue's accesses to 8-bit rows in global memory, against the CPU oracle, bit-exact: pitches, offsets
and pointers on the 16-byte grid but off the 32-byte one, odd numbers of 16-column chunks, residual rows of another alignment
than the output's, one tile and several per CTA, CTA pairs; bytes beside the rows untouched."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8 = 0, 1

CASES = [
    # name, N,H,W,C,K,R,pad, y type, residual, pitch - K, channel offset, output shift, residual shift (bytes)
    ("k16", 2, 20, 21, 64, 16, 3, 1, U8, True, 0, 0, 0, 0),
    ("k48_odd_chunks", 3, 45, 45, 64, 48, 1, 0, U8, True, 0, 0, 0, 0),
    ("k64_slice_16", 4, 33, 33, 64, 64, 1, 0, U8, True, 32, 16, 0, 0),
    ("k64_pitch_80", 4, 60, 60, 64, 64, 3, 1, S8, True, 16, 0, 0, 0),
    ("k96_output_off", 2, 30, 31, 96, 96, 3, 1, U8, True, 0, 0, 16, 0),
    ("k96_residual_off", 2, 30, 31, 96, 96, 3, 1, U8, True, 0, 0, 0, 16),
    ("k112_short", 1, 14, 14, 320, 112, 1, 0, U8, True, 16, 0, 0, 0),
    ("k208_long", 16, 57, 57, 64, 208, 1, 0, S8, True, 0, 0, 0, 0),
    ("k256_one_tile_a_cta", 8, 28, 28, 256, 256, 3, 1, U8, True, 0, 0, 0, 0),
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
