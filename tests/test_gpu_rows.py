"""GPU parity of tensor-core layers whose 8-bit output or residual rows are off the 16-byte grid (their rows are moved by
the epilogue warps), against the CPU oracle, bit-exact: channel counts around the words of a row and the widths of a
tile, slices at odd offsets, unaligned pointers, one and several tiles per CTA, halo and plain tiles; bytes beside the
rows untouched."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8 = 0, 1

CASES = [
    # name, N,H,W,C,K,R,S,stride,pad, y type, residual, per channel, pitch - K, channel offset, pointer offset
    ("k1", 2, 30, 31, 64, 1, 3, 3, 1, (1, 1), U8, True, False, 0, 0, 0),
    ("k7_5x5", 2, 40, 40, 16, 7, 5, 5, 1, (2, 2), S8, True, True, 0, 0, 0),
    ("k33", 3, 45, 45, 64, 33, 1, 1, 1, (0, 0), U8, True, False, 0, 0, 0),
    ("k60_strided", 2, 57, 57, 64, 60, 1, 1, 2, (0, 0), U8, False, False, 0, 0, 0),
    ("k100_halo_long", 32, 56, 56, 32, 100, 3, 3, 1, (1, 1), U8, True, False, 0, 0, 0),
    ("k250_long", 16, 57, 57, 64, 250, 1, 1, 1, (0, 0), S8, True, False, 0, 0, 0),
    ("k250_shared_tile", 4, 28, 28, 640, 250, 1, 1, 1, (0, 0), U8, True, True, 0, 0, 0),
    ("k500_two_tiles", 6, 28, 28, 320, 500, 3, 3, 1, (1, 1), U8, False, False, 0, 0, 0),
    ("k301_narrow", 1, 14, 14, 1024, 301, 1, 1, 1, (0, 0), U8, True, False, 0, 0, 0),
    ("k256_odd_slice", 4, 33, 33, 128, 256, 1, 1, 1, (0, 0), U8, True, False, 13, 6, 1),
    ("k61_pairs_of_pixels", 2, 30, 240, 16, 61, 7, 7, 2, (3, 3), U8, False, True, 3, 2, 3),
    # rows on the grid that end off it: the channels up to the next 16-byte line belong to somebody else
    ("k24_of_48", 2, 33, 33, 64, 24, 1, 1, 1, (0, 0), U8, False, False, 24, 0, 0),
    ("k88_of_128_halo", 2, 40, 40, 32, 88, 3, 3, 1, (1, 1), S8, False, True, 40, 16, 0),
    ("k3_of_16_long", 4, 80, 80, 64, 3, 3, 3, 1, (1, 1), U8, False, False, 13, 0, 0),
    ("k24_slice_aligned_pitch", 2, 33, 33, 64, 24, 1, 1, 1, (0, 0), U8, True, False, 24, 16, 0),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_rows_off_the_grid_match_oracle(q8, case):
    name, N, H, W, C, K, R, S, st, pad, ytype, res, per_channel, extra, c_off, shift = case
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, S, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, (st, st), pad, (1, 1), threads=8)
    P, Q = acc.shape[1:3]
    resid = g.integers(0, 256, acc.shape, dtype=np.uint8) if res else None
    scale = (g.uniform(0.5, 1.5, K if per_channel else 1) * 100.0 / max(1, np.abs(acc).max())).astype(np.float32)
    want = o.epilogue(acc, scale if per_channel else scale[0], resid, 0.37 if res else 0.0, ytype == U8, o.U8 if ytype == U8 else o.S8)
    ldc = K + extra
    d = q8.make_conv_desc(N, H, W, C, K, R, S, (st, st), pad, (1, 1), U8, U8, ytype, ytype == U8, K if per_channel else 1, ldc, c_off)
    plan = q8.q8_conv2d_query_plan(d, res)
    assert plan.kernel == q8.Q8_KERNEL_TMA and plan.moved_rows
    assert plan.shared_groups == (4 if name in ("k250_shared_tile", "k60_strided", "k500_two_tiles", "k256_odd_slice", "k61_pairs_of_pixels", "k88_of_128_halo") else 1)
    assert plan.operand == (1 if "strided" in name else (2 if R > 1 else 0))
    rows = N * P * Q
    buf = torch.full((64 + rows * ldc + 64,), 7, dtype=q8.TORCH_DTYPES[ytype], device="cuda")
    y = buf[64 + shift:64 + shift + rows * ldc].view(N, P, Q, ldc)
    rbuf = torch.zeros(rows * K + 3, dtype=torch.uint8, device="cuda")
    rd = None
    if res:
        rd = rbuf[shift:shift + rows * K].view(N, P, Q, K)
        rd.copy_(torch.from_numpy(resid).cuda())
    args = [torch.from_numpy(a).cuda() for a in (x, w, bias, scale)]
    algos = [q8.Q8_ALGO_AUTO] + [q8.Q8_ALGO_UMMA] * (ldc % 16 == 0 and c_off % 16 == 0 and shift == 0)
    for d.algo in algos:
        buf.fill_(7)
        q8.q8_conv2d(d, *args, rd, 0.37 if res else 0.0, y)
        q8.q8_read_status()
        got = y.cpu().numpy()
        assert np.array_equal(got[..., c_off:c_off + K], want)
        assert (got[..., :c_off] == 7).all() and (got[..., c_off + K:] == 7).all()
        assert bool((buf[:64 + shift] == 7).all()) and bool((buf[64 + shift + rows * ldc:] == 7).all())
