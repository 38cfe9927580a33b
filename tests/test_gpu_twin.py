"""GPU parity of layers whose CTAs run two tiles at once on one pass of the weights (between one and two tiles per SM, streamed
weights, one tile of columns), against the CPU oracle, bit-exact: odd numbers of tiles, last channel blocks of one, two and
three K steps, moved rows, residual sums, 32-bit outputs, dilation."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8, S32, F32 = 0, 1, 2, 3
OT = {U8: o.U8, S8: o.S8, S32: o.S32, F32: o.F32}

CASES = [
    # name, N,H,W,C,K,R,S,pad,dil, y type, residual
    ("1x7_c160", 38, 17, 17, 160, 160, 1, 7, (0, 3), 1, U8, True),
    ("7x1_c208_odd", 51, 17, 17, 208, 144, 7, 1, (3, 0), 1, S8, False),
    ("3x3_c224_k192", 50, 14, 21, 224, 192, 3, 3, (1, 1), 1, U8, True),
    ("3x3_c128_k180_rows", 151, 9, 12, 128, 180, 3, 3, (1, 1), 1, U8, True),
    ("3x3_c160_f32", 149, 9, 12, 160, 172, 3, 3, (1, 1), 1, F32, False),
    ("3x3_c64_k160_raw", 150, 9, 12, 64, 160, 3, 3, (1, 1), 1, S32, False),
    ("3x3_c128_k192_dil2", 75, 14, 14, 128, 192, 3, 3, (2, 2), 2, U8, True),
    ("3x3_c96_k176", 150, 9, 12, 96, 176, 3, 3, (1, 1), 1, U8, False),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_twin_tiles_match_oracle(q8, case):
    name, N, H, W, C, K, R, S, pad, dil, ytype, res = case
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, S, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, (1, 1), pad, (dil, dil), threads=16)
    resid = g.integers(0, 256, acc.shape, dtype=np.uint8) if res else None
    scale = np.float32(100.0 / max(1, np.abs(acc).max()))
    want = o.epilogue(acc, scale, resid, 0.37 if res else 0.0, ytype != S8, OT[ytype])
    d = q8.make_conv_desc(N, H, W, C, K, R, S, (1, 1), pad, (dil, dil), U8, U8, ytype, ytype != S8)
    plan = q8.q8_conv2d_query_plan(d, res)
    assert plan.kernel == q8.Q8_KERNEL_TMA and plan.operand == 2 and plan.weights == 2 and not plan.cta_pair
    y = torch.full(acc.shape, 7, dtype=q8.TORCH_DTYPES[ytype], device="cuda")
    q8.q8_conv2d(d, torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), torch.from_numpy(bias).cuda(),
                 torch.tensor([scale], device="cuda"), torch.from_numpy(resid).cuda() if res else None, 0.37 if res else 0.0, y)
    q8.q8_read_status()
    assert np.array_equal(y.cpu().numpy().view(np.uint8), np.ascontiguousarray(want).view(np.uint8))
