"""GPU parity of the tensor-core convolution that packs rows of three-channel images, against the CPU oracle, bit-exact: every
run length and number of runs, one and several K blocks, tiles across image ends, padding on all sides, dilation along H,
inputs and residuals off the 16-byte grid, slices of wider outputs, channel counts off the 16-column chunks, every output type
with and without a residual, one multiplier and one per channel.  Filters of one row and several columns are gathered."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8, S32, F32 = 0, 1, 2, 3
OT = {U8: o.U8, S8: o.S8, S32: o.S32, F32: o.F32}

CASES = [
    # name, N,H,W,C,K,R,S,strides,pads,dil_h, x signed, y type, residual, per channel, extra channels per pixel, input shift
    ("c3_3x3s2", 5, 99, 97, 3, 32, 3, 3, (2, 2), (0, 0), 1, True, U8, False, False, 0, 0),
    ("c3_3x3_pad", 8, 40, 37, 3, 64, 3, 3, (1, 1), (1, 1), 1, True, U8, True, False, 0, 1),
    ("c3_7x7s2_pad3", 11, 64, 62, 3, 64, 7, 7, (2, 2), (3, 3), 1, True, S8, False, True, 0, 2),
    ("c3_5x5_k128", 11, 30, 31, 3, 128, 5, 5, (1, 1), (2, 2), 1, False, U8, True, False, 0, 0),
    ("c3_1x7_f32", 8, 33, 40, 3, 24, 1, 7, (1, 1), (0, 3), 1, False, F32, True, True, 0, 3),
    ("c3_7x1_runs_of_three", 8, 33, 40, 3, 80, 7, 1, (1, 1), (3, 0), 1, False, U8, False, False, 32, 0),
    ("c3_1x1", 12, 30, 30, 3, 8, 1, 1, (1, 1), (0, 0), 1, False, S32, False, False, 0, 1),
    ("c3_3x5_strides_3_1", 50, 26, 24, 3, 32, 3, 5, (3, 1), (2, 0), 1, False, U8, False, False, 0, 0),
    ("c3_5x3_dil_h2", 26, 30, 29, 3, 48, 5, 3, (1, 2), (2, 1), 2, False, U8, False, False, 0, 0),
    ("c3_7x3_s8_residual", 32, 17, 18, 3, 48, 7, 3, (1, 1), (3, 1), 1, True, S8, True, False, 0, 0),
    ("c3_1x5", 16, 16, 40, 3, 112, 1, 5, (1, 1), (0, 2), 1, False, U8, False, False, 0, 1),
    ("c3_5x7", 30, 21, 22, 3, 96, 5, 7, (1, 1), (0, 3), 1, True, U8, False, True, 32, 2),
    ("many_tiles_c3", 8, 150, 150, 3, 32, 3, 3, (1, 1), (1, 1), 1, True, U8, False, False, 0, 0),
    ("wide_padding", 13, 14, 14, 3, 16, 3, 3, (1, 1), (7, 9), 1, True, U8, False, False, 0, 0),
    ("c3_3x3_f32", 6, 45, 47, 3, 36, 3, 3, (1, 1), (1, 1), 1, True, F32, False, False, 8, 2),
    ("c3_7x7s2_f32_residual", 11, 64, 62, 3, 64, 7, 7, (2, 2), (3, 3), 1, False, F32, True, False, 0, 0),
    ("c3_5x5_f32_per_channel", 11, 31, 30, 3, 112, 5, 5, (1, 1), (2, 2), 1, True, F32, False, True, 0, 1),
    ("c3_3x1_f32_residual_off_per_channel", 12, 33, 40, 3, 44, 3, 1, (1, 1), (1, 0), 1, True, F32, True, True, 8, 0),
    ("c3_3x3_s32", 6, 45, 47, 3, 20, 3, 3, (1, 1), (1, 1), 1, True, S32, False, False, 8, 0),
    ("c3_3x3_s32_k52", 6, 45, 47, 3, 52, 3, 3, (1, 1), (1, 1), 1, False, S32, False, False, 0, 1),
    ("c3_3x3_residual_off", 8, 40, 37, 3, 48, 3, 3, (1, 1), (1, 1), 1, True, U8, True, False, 32, 0),
    ("c3_7x7s2_s8_residual_off", 9, 64, 66, 3, 32, 7, 7, (2, 2), (3, 3), 1, False, S8, True, True, 0, 3),
]
GATHERED = ("c3_1x7_f32", "c3_1x5")


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_packed_matches_oracle(q8, case):
    name, N, H, W, C, K, R, S, st, pad, dil_h, xs8, ytype, res, per_channel, extra, shift = case
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(-128, 128, (N, H, W, C)).astype(np.int8) if xs8 else g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, S, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, st, pad, (dil_h, 1), threads=8)
    P, Q = acc.shape[1:3]
    resid = g.integers(0, 256, (N, P, Q, K), dtype=np.uint8) if res else None
    scale = (g.uniform(0.5, 1.5, K if per_channel else 1) * 100.0 / max(1, np.abs(acc).max())).astype(np.float32)
    want = o.epilogue(acc, scale if per_channel else scale[0], resid, 0.37 if res else 0.0, True, OT[ytype])
    d = q8.make_conv_desc(N, H, W, C, K, R, S, st, pad, (dil_h, 1), S8 if xs8 else U8, U8, ytype, True,
                          K if per_channel else 1, K + extra, extra // 2)
    plan = q8.q8_conv2d_query_plan(d, res)
    assert plan.kernel == q8.Q8_KERNEL_GATHER and plan.operand == (0 if name in GATHERED else 3)
    xb = torch.zeros(x.size + 3, dtype=torch.uint8, device="cuda")
    xb[shift:shift + x.size] = torch.from_numpy(x.view(np.uint8).ravel()).cuda()
    rd, off = None, 1 if "residual_off" in name else 0
    if res:
        rb = torch.zeros(resid.size + 1, dtype=torch.uint8, device="cuda")
        rd = rb[off:off + resid.size].view(N, P, Q, K)
        rd.copy_(torch.from_numpy(resid).cuda())
    y = torch.full((N, P, Q, K + extra), 7, dtype=q8.TORCH_DTYPES[ytype], device="cuda")
    q8.q8_conv2d(d, xb[shift:shift + x.size].view(N, H, W, C), torch.from_numpy(w).cuda(), torch.from_numpy(bias).cuda(),
                 torch.from_numpy(scale).cuda(), rd, 0.37 if res else 0.0, y)
    q8.q8_read_status()
    got = y.cpu().numpy()
    lo, hi = extra // 2, extra // 2 + K
    a, e = np.ascontiguousarray(got[..., lo:hi]), want
    if ytype == F32:
        a, e = a.view(np.uint32), e.view(np.uint32)
    assert np.array_equal(a, e)
    assert (got[..., :lo] == 7).all() and (got[..., hi:] == 7).all()   # neighbours of the slice untouched
