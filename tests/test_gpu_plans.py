"""GPU parity of the launch plans that a layer's size selects, against the CPU oracle, bit-exact: narrow column tiles of
every width, and CTA pairs whose epilogue groups share a tile's columns, both with one multiplier per channel."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu
U8, S8 = 0, 1

CASES = [
    # name, N,H,W,C,K,R,S,pad, y type, residual, tile width, CTA pair, groups that share a tile's columns
    ("narrow_16", 1, 14, 14, 1024, 256, 1, 1, (0, 0), U8, True, 16, 0, 1),
    ("narrow_16_halo", 1, 7, 7, 512, 512, 3, 3, (1, 1), S8, False, 16, 0, 1),
    ("narrow_32_ragged", 4, 14, 14, 640, 528, 1, 1, (0, 0), U8, True, 32, 0, 1),
    ("narrow_32_short_reduction", 1, 7, 7, 512, 2048, 1, 1, (0, 0), U8, True, 32, 0, 1),
    ("narrow_64_ragged", 4, 14, 14, 576, 1008, 1, 1, (0, 0), S8, False, 64, 0, 4),
    ("narrow_128", 16, 14, 14, 768, 512, 1, 1, (0, 0), U8, False, 128, 0, 4),
    ("pair_256_shared", 14, 53, 53, 128, 512, 3, 3, (1, 1), U8, True, 256, 1, 2),
    ("pair_160_five_chunks_a_group", 44, 37, 37, 128, 160, 3, 3, (1, 1), S8, False, 160, 1, 2),
    ("pair_224_seven_chunks_a_group", 30, 37, 37, 96, 224, 3, 3, (1, 1), S8, True, 224, 1, 2),
    ("pair_96_alone", 44, 37, 37, 128, 96, 3, 3, (1, 1), U8, False, 96, 1, 1),
    ("wide_144_single_cta", 44, 37, 37, 128, 144, 3, 3, (1, 1), S8, False, 144, 0, 1),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_plan_matches_oracle(q8, case):
    name, N, H, W, C, K, R, S, pad, ytype, res, tile_n, pair, shared = case
    g = np.random.default_rng(sum(map(ord, name)))
    x = g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, R, S, C)).astype(np.int8)
    bias = g.integers(-5000, 5000, K).astype(np.int32)
    acc = o.conv_acc(x, w, bias, (1, 1), pad, (1, 1), threads=8)
    resid = g.integers(0, 256, acc.shape, dtype=np.uint8) if res else None
    scale = (g.uniform(0.5, 1.5, K) * 100.0 / max(1, np.abs(acc).max())).astype(np.float32)
    want = o.epilogue(acc, scale, resid, 0.37 if res else 0.0, ytype == U8, o.U8 if ytype == U8 else o.S8)
    d = q8.make_conv_desc(N, H, W, C, K, R, S, (1, 1), pad, (1, 1), U8, U8, ytype, ytype == U8, K)
    plan = q8.q8_conv2d_query_plan(d, res)
    assert (plan.kernel, plan.tile_n, plan.cta_pair, plan.shared_groups) == (q8.Q8_KERNEL_TMA, tile_n, pair, shared)
    args = [torch.from_numpy(a).cuda() for a in (x, w, bias, scale)]
    rd = torch.from_numpy(resid).cuda() if res else None
    for _ in range(2):   # twice: the second launch follows the first in the stream
        y = q8.q8_conv2d(d, *args, rd, 0.37 if res else 0.0)
    q8.q8_read_status()
    assert np.array_equal(y.cpu().numpy(), want)


@pytest.mark.parametrize("K", [32, 33])
@pytest.mark.parametrize("ytype", [U8, S8])
def test_layer_that_no_tile_of_the_tma_fed_kernel_fits(q8, K, ytype):
    """Filter rows 70 apart with stride 2: a halo patch exceeds shared memory, and im2col maps end at 128 rows."""
    g = np.random.default_rng(K)
    x = g.integers(0, 256, (1, 200, 128, 16), dtype=np.uint8)
    w = g.integers(-128, 128, (K, 3, 1, 16)).astype(np.int8)
    scale = np.float32(1e-3)
    want = o.conv2d(x, w, None, scale, stride=(2, 1), dil=(70, 1), relu=True, y_type=o.U8 if ytype == U8 else o.S8, threads=8)
    d = q8.make_conv_desc(1, 200, 128, 16, K, 3, 1, (2, 1), (0, 0), (70, 1), U8, U8, ytype, True)
    args = [torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), None, torch.tensor([scale], device="cuda")]
    y = q8.q8_conv2d(d, *args)
    q8.q8_read_status()
    assert np.array_equal(y.cpu().numpy(), want)
    d.algo = q8.Q8_ALGO_UMMA
    with pytest.raises(q8.Q8Error) as e:
        q8.q8_conv2d(d, *args)
    assert e.value.code == 2


@pytest.mark.parametrize("shape", [(2, 95, 198, 32, 8, 3), (2, 95, 198, 32, 16, 3), (1, 60, 60, 32, 32, 9), (1, 95, 60, 64, 48, 6)],
                         ids=lambda s: "x".join(map(str, s)))
def test_pixel_pairs_whose_patch_does_not_fit(q8, shape):
    """Stride-2 filters of tall dilated columns: the patch of pixel pairs exceeds shared memory."""
    N, H, W, C, K, dil = shape
    g = np.random.default_rng(K)
    x = g.integers(0, 256, (N, H, W, C), dtype=np.uint8)
    w = g.integers(-128, 128, (K, 7, 1, C)).astype(np.int8)
    scale = np.float32(4e-4)
    want = o.conv2d(x, w, None, scale, stride=(2, 2), pad=(2, 0), dil=(dil, 1), relu=True, y_type=o.U8, threads=8)
    d = q8.make_conv_desc(N, H, W, C, K, 7, 1, (2, 2), (2, 0), (dil, 1), U8, U8, U8, True)
    y = q8.q8_conv2d(d, torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), None, torch.tensor([scale], device="cuda"))
    q8.q8_read_status()
    assert np.array_equal(y.cpu().numpy(), want)
