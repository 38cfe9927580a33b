"""GPU parity of the gathering tensor-core convolution (channel counts off the 16-channel grid, unaligned operands)
against the CPU oracle, bit-exact: one and several K blocks of every block width, runs that end inside a chunk, column
tiles with a ragged tail, weights resident and streamed, every output type."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8, S32, F32 = 0, 1, 2, 3
OT = {U8: o.U8, S8: o.S8, S32: o.S32, F32: o.F32}

CASES = [
    # name, N,H,W,C,K,R,S,stride,pad,dil, x signed, y type, residual, per channel, extra channels per pixel
    ("one_chunk_pair_c20_1x1", 12, 60, 60, 20, 33, 1, 1, 1, (0, 0), 1, False, U8, True, False, 0),
    ("three_chunks_c3_3x3s2", 2, 61, 59, 3, 32, 3, 3, 2, (0, 0), 1, True, U8, False, False, 0),
    ("c3_7x7s2_pad3", 2, 64, 62, 3, 64, 7, 7, 2, (3, 3), 1, True, S8, False, True, 0),
    ("c1_5x5_k1_raw", 3, 20, 21, 1, 1, 5, 5, 1, (2, 2), 1, False, S32, False, False, 0),
    ("c100_3x3_k130_two_column_tiles", 1, 12, 11, 100, 130, 3, 3, 1, (1, 1), 1, False, U8, True, True, 0),
    ("c17_dil2_f32", 2, 15, 14, 17, 24, 3, 3, 1, (2, 2), 2, False, F32, False, False, 0),
    ("c5_1x7_slice", 6, 39, 60, 5, 21, 1, 7, 1, (0, 3), 1, True, U8, False, False, 13),
    ("resident_weights_many_tiles_c12", 2, 110, 100, 12, 40, 3, 3, 1, (1, 1), 1, False, U8, False, False, 0),
    ("stride9_c16", 1, 40, 40, 16, 16, 3, 3, 9, (1, 1), 1, False, U8, False, False, 0),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_gather_matches_oracle(q8, case):
    name, N, H, W, C, K, R, S, st, pad, dil, xs8, ytype, res, per_channel, extra = case
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(-128, 128, (N, H, W, C)).astype(np.int8) if xs8 else g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, S, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, (st, st), pad, (dil, dil), threads=8)
    P, Q = acc.shape[1:3]
    resid = g.integers(0, 256, (N, P, Q, K), dtype=np.uint8) if res else None
    scale = (g.uniform(0.5, 1.5, K if per_channel else 1) * 100.0 / max(1, np.abs(acc).max())).astype(np.float32)
    want = o.epilogue(acc, scale if per_channel else scale[0], resid, 0.37 if res else 0.0, True, OT[ytype])
    d = q8.make_conv_desc(N, H, W, C, K, R, S, (st, st), pad, (dil, dil), S8 if xs8 else U8, U8, ytype, True,
                          K if per_channel else 1, K + extra, extra // 2)
    assert q8.q8_conv2d_query_plan(d, res).kernel == q8.Q8_KERNEL_GATHER
    xb = torch.zeros(x.size + 1, dtype=torch.uint8, device="cuda")   # input one byte off the allocation's alignment
    xb[1:] = torch.from_numpy(x.view(np.uint8).ravel()).cuda()
    y = torch.full((N, P, Q, K + extra), 7, dtype=q8.TORCH_DTYPES[ytype], device="cuda")
    q8.q8_conv2d(d, xb[1:].view(N, H, W, C), torch.from_numpy(w).cuda(), torch.from_numpy(bias).cuda(), torch.from_numpy(scale).cuda(),
                 torch.from_numpy(resid).cuda() if res else None, 0.37 if res else 0.0, y)
    q8.q8_read_status()
    got = y.cpu().numpy()
    lo, hi = extra // 2, extra // 2 + K
    a, e = np.ascontiguousarray(got[..., lo:hi]), want
    if ytype == F32:
        a, e = a.view(np.uint32), e.view(np.uint32)
    assert np.array_equal(a, e)
    assert (got[..., :lo] == 7).all() and (got[..., hi:] == 7).all()   # neighbours of the slice untouched
