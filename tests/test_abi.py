"""CPU checks of the C ABI: the library loads, exports what include/q8.h declares, and its host-side
validation turns bad requests into documented error codes without launching anything."""
import ctypes as C
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import oracle as o
import paper_1805_08691_b200 as q8

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "q8.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(q8_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported_and_bound():
    names = _declared()
    assert len(names) >= 18
    for n in names:
        assert hasattr(q8.lib, n), n
        assert n in q8.EXPORTS, n
        assert callable(getattr(q8, n)), n  # the Python binding carries the same name


def test_struct_layout_matches_header():
    text = open(os.path.join(ROOT, "include", "q8.h")).read()
    body = re.search(r"typedef struct q8_conv_desc \{(.*?)\} q8_conv_desc;", text, flags=re.S).group(1)
    body = re.sub(r"/\*.*?\*/", "", body, flags=re.S)
    fields = []
    for decl in body.split(";"):
        decl = decl.strip()
        if decl.startswith("int32_t"):
            fields += [f.strip() for f in decl[len("int32_t"):].split(",")]
    assert fields == [f[0] for f in q8.q8_conv_desc._fields_]
    assert C.sizeof(q8.q8_conv_desc) == 4 * len(fields)


def test_host_helpers_agree_with_oracle():
    g = np.random.default_rng(0)
    for _ in range(2000):
        m = float(np.float32(g.uniform(1e-4, 1e4)))
        for p in (7, 8):
            assert q8.q8_factor(m, p) == o.factor(m, p)
        a, b, c = (float(np.float32(v)) for v in g.uniform(1e-4, 1.0, 3))
        assert q8.q8_requant_scale(a, b, c) == o.requant_scale(a, b, c)
        assert q8.q8_bias_factor(a, b) == o.bias_factor(a, b)
    assert q8.q8_factor(0.0, 8) == 1.0
    for H, k, st, pad, ceil in [(75, 2, 2, 0, True), (75, 2, 2, 0, False), (112, 3, 2, 1, False), (147, 3, 2, 0, False),
                                (8, 8, 1, 0, False), (19, 3, 1, 1, False)]:
        assert q8.q8_pool_out_extent(H, k, st, pad, ceil) == o.pool_out(H, k, st, pad, ceil)


def _code(fn, *a, **k):
    with pytest.raises(q8.Q8Error) as e:
        fn(*a, **k)
    return e.value.code


def test_bad_requests_are_rejected_on_the_host():
    assert _code(q8.q8_factor, float("nan"), 8) == 7
    assert _code(q8.q8_factor, float("inf"), 8) == 7
    assert _code(q8.q8_factor, 1.0, 0) == 1
    assert _code(q8.q8_requant_scale, 0.0, 1.0, 1.0) == 7
    d = q8.make_conv_desc(1, 8, 8, 16, 16, 3, 3)
    assert q8.q8_conv2d_workspace_bytes(d) == 0
    for field, bad in [("N", 0), ("C", -1), ("stride_h", 0), ("pad_w", -1), ("x_type", 3), ("y_type", 9),
                       ("scale_count", 2), ("algo", 5), ("y_ldc", 8), ("y_c_offset", -16)]:
        d = q8.make_conv_desc(1, 8, 8, 16, 16, 3, 3)
        setattr(d, field, bad)
        assert _code(q8.q8_conv2d_query_algo, d) == 1, field
    # filter larger than the padded image -> empty output
    assert _code(q8.q8_conv2d_query_algo, q8.make_conv_desc(1, 2, 2, 16, 16, 3, 3)) == 1
    # accumulator overflow guard
    assert _code(q8.q8_conv2d_query_algo, q8.make_conv_desc(1, 16, 16, 8192, 16, 3, 3)) == 1
    # null pointers never reach a launch
    d = q8.make_conv_desc(1, 8, 8, 16, 16, 3, 3)
    rc = q8.lib.q8_conv2d(C.byref(d), None, None, None, None, None, 0.0, None, None, 0, None)
    assert rc == 1 and b"null" in q8.lib.q8_last_error()
    assert q8.lib.q8_quantize(None, 10, 1.0, 0, None, None) == 1
    assert q8.lib.q8_quantize(None, 0, 0.0, 0, None, None) == 7
    assert q8.lib.q8_calibrate_maxabs(None, 4, None, None) == 1
    assert q8.lib.q8_dequantize(None, 3, 4, 1.0, None, None) == 1
    assert q8.lib.q8_fold_bn(None, None, None, None, None, None, 1e-5, 4, 4, None, None, None) == 1


def test_kernel_selection_rules():
    U = q8.Q8_ALGO_UMMA
    assert q8.q8_conv2d_query_algo(q8.make_conv_desc(32, 56, 56, 256, 64, 1, 1)) == U
    assert q8.q8_conv2d_query_algo(q8.make_conv_desc(32, 56, 56, 64, 64, 3, 3, pad=(1, 1))) == U
    assert q8.q8_conv2d_query_algo(q8.make_conv_desc(1, 8, 8, 3, 8, 3, 3, pad=(1, 1))) == q8.Q8_ALGO_DIRECT
    assert q8.q8_conv2d_query_algo(q8.make_conv_desc(32, 56, 56, 64, 64, 3, 3, pad=(1, 1), algo=q8.Q8_ALGO_DIRECT)) == q8.Q8_ALGO_DIRECT


D, G, T = q8.Q8_KERNEL_DIRECT, q8.Q8_KERNEL_GATHER, q8.Q8_KERNEL_TMA
U8, S8, S32, F32 = q8.Q8_U8, q8.Q8_S8, q8.Q8_S32, q8.Q8_F32

ROUTES = [
    # kernel, N,H,W,C,K,R,S, further descriptor fields
    (T, 32, 56, 56, 64, 64, 3, 3, dict(pad=(1, 1))),
    (T, 32, 56, 56, 64, 250, 1, 1, {}),                                # 8-bit rows off the 16-byte grid: moved by the warps
    (T, 32, 56, 56, 64, 256, 1, 1, dict(y_ldc=300, y_c_offset=13)),
    (G, 1, 56, 56, 64, 9, 1, 1, {}),                                   # ... unless short, with a short reduction
    (T, 1, 56, 56, 64, 9, 1, 1, dict(y_type=F32)),
    (D, 1, 8, 8, 16, 9, 1, 1, {}),                                     # ... or tiny
    (T, 1, 8, 8, 16, 16, 1, 1, {}),
    (G, 2, 28, 28, 100, 120, 3, 3, dict(pad=(1, 1))),
    (D, 1, 8, 8, 3, 8, 1, 1, {}),
    (D, 2, 9, 9, 16, 5000, 1, 1, {}),
    (G, 8, 299, 299, 3, 32, 3, 3, dict(stride=(2, 2))),
    (D, 1, 1, 1, 163, 397, 7, 7, dict(pad=(3, 3))),                    # few outputs or few products: no tensor cores
    (D, 7, 1, 1, 64, 9, 7, 7, dict(pad=(3, 3), stride=(2, 2))),
    (D, 9, 160, 160, 5, 1, 1, 1, {}),
    (D, 1, 31, 9, 2, 444, 1, 1, {}),
    (D, 1, 9, 12, 32, 44, 1, 1, {}),
    (G, 1, 200, 128, 16, 32, 3, 1, dict(stride=(2, 1), dil=(70, 1))),  # no tile fits
    (G, 1, 60, 60, 32, 32, 7, 1, dict(stride=(2, 2), pad=(2, 0), dil=(9, 1))),   # nor in whole pixel pairs
    (G, 1, 1, 1 << 19, 1025, 8, 1, 1, dict(stride=(1, 1 << 14))),
    (D, 1, 1, 1 << 21, 1025, 8, 1, 1, dict(stride=(1, 1 << 17))),      # rows of more than 2^30 bytes, with and
    (D, 1, 1, 1000, 1025, 8, 1, 1, dict(stride=(1, 1 << 17), pad=(0, 1 << 20))),   # without their padding
    (D, 1, 300, 8, 5, 64, 2, 2, dict(dil=(1 << 28, 1), pad=(1 << 27, 0))),        # filter rows 2^28 apart
]


@pytest.mark.parametrize("route", ROUTES, ids=lambda r: "x".join(map(str, r[1:8])) + "".join(f"_{v}" for v in r[8].values()))
def test_queries_follow_the_dispatch(route):
    kernel, fields, more = route[0], route[1:8], route[8]
    d = q8.make_conv_desc(*fields, **more)
    assert q8.q8_conv2d_query_plan(d).kernel == kernel
    assert (q8.q8_conv2d_query_algo(d) == q8.Q8_ALGO_UMMA) == (kernel == T)
    d.algo = q8.Q8_ALGO_DIRECT
    assert q8.q8_conv2d_query_plan(d).kernel == D and q8.q8_conv2d_query_algo(d) == q8.Q8_ALGO_DIRECT
    # asked for by name, the TMA-fed kernel also refuses rows off the grid
    d.algo = q8.Q8_ALGO_UMMA
    ldc = d.y_ldc or d.K
    if kernel == T and (d.y_type == F32 or (ldc % 16 == 0 and d.y_c_offset % 16 == 0)):
        assert q8.q8_conv2d_query_plan(d).kernel == T and q8.q8_conv2d_query_algo(d) == q8.Q8_ALGO_UMMA
    elif kernel == T or d.C % 16 or d.K > 4096 or d.y_type in (U8, S8):
        assert q8.q8_conv2d_query_algo(d) == q8.Q8_ALGO_DIRECT
        assert _code(q8.q8_conv2d_query_plan, d) == 2


@pytest.mark.parametrize("K", [8, 16])
def test_pixel_pairs_are_never_cut_into_channel_blocks(K):
    """A patch of whole 64-byte pixel pairs does not fit here: the layer takes im2col loads, not narrower blocks of pairs."""
    d = q8.make_conv_desc(2, 95, 198, 32, K, 7, 1, (2, 2), (2, 0), (3, 1))
    plan = q8.q8_conv2d_query_plan(d)
    assert (plan.kernel, plan.operand) == (T, 1)


@pytest.mark.parametrize("shape,parts", [((64, 1, 1, 8192, 1008, 1, 1), 16), ((64, 1, 1, 2048, 1008, 1, 1), 1), ((1, 14, 14, 1024, 256, 1, 1), 1),
                                         ((1, 64, 74, 2048, 256, 1, 1), 1), ((8, 7, 7, 6144, 512, 1, 1), 12), ((2, 10, 10, 8192, 9, 1, 1), 1)])
def test_scratch_is_asked_for_by_the_layers_that_split(shape, parts):
    d = q8.make_conv_desc(*shape)
    assert q8.q8_conv2d_query_plan(d).splits == parts
    assert q8.q8_conv2d_workspace_bytes(d) == (parts * shape[0] * shape[1] * shape[2] * shape[4] * 4 if parts > 1 else 0)
    d.y_type, d.relu = S32, 0
    assert q8.q8_conv2d_workspace_bytes(d) == 0


@pytest.mark.parametrize("name", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_private_torch_entry_points_are_optional(name):
    code = (f"import torch; delattr(torch._C, {name!r}); import types; import paper_1805_08691_b200.binding as b; "
            "torch.cuda.is_initialized = lambda: True; torch.cuda.current_stream = lambda: types.SimpleNamespace(cuda_stream=77); "
            "assert b._stream() == 77")
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT)


def test_recording_requests_are_checked_on_the_host():
    assert _code(q8.q8_record_begin, 0) == 1
    assert q8.lib.q8_record_replay(None, None) == 1
    assert q8.lib.q8_record_end(1, (C.c_void_p * 1)(), None) == 1
    q8.q8_record_free(None)


def test_marshalled_calls_refuse_what_they_cannot_pass():
    """Host tensors, views and objects that are no tensors are refused with the argument's name, before any call."""
    import torch
    d = q8.make_conv_desc(1, 4, 4, 16, 16, 1, 1)
    x = torch.zeros((1, 4, 4, 16), dtype=torch.uint8)
    w, y = torch.zeros((16, 1, 1, 16), dtype=torch.int8), torch.zeros((1, 4, 4, 16), dtype=torch.uint8)
    for bad in (x, x.permute(0, 2, 1, 3), 3, [1]):
        with pytest.raises(TypeError, match="^x: expected a contiguous CUDA tensor"):
            q8.q8_conv2d(d, bad, w, None, None, y=y)
    for no_desc in (q8.q8_conv_plan(), bytes(d), bytearray(d), C.byref(d)):
        with pytest.raises(TypeError, match="q8_conv_desc"):
            q8.q8_conv2d(no_desc, x, w, None, None, y=y)

    class wider(q8.q8_conv_desc):
        _fields_ = [("note", C.c_int32)]
    with pytest.raises(TypeError, match="^x: expected"):   # a derived structure is one
        q8.q8_conv2d(wider(*bytes(21)), x, w, None, None, y=y)
    with pytest.raises(TypeError, match="^out: expected|^x: expected"):
        q8.q8_quantize(torch.zeros(4), 1.0, q8.Q8_U8)
    with pytest.raises(TypeError, match="^loc: expected a CUDA fp32 tensor"):
        q8.q8_detection_output([(torch.zeros(1, 4, 4), torch.zeros(1, 4, 3), 1)], torch.zeros(4, 4), (0.1,) * 4, 3,
                               workspace=torch.zeros(1, dtype=torch.uint8), out=torch.zeros(1), counts=torch.zeros(1))


@pytest.mark.parametrize("N,HW,C,K,R,residual,buffers", [
    (64, 56, 64, 256, 1, True, 8), (64, 56, 64, 256, 1, False, 8),     # the expanding layers of early residual blocks
    (64, 28, 128, 512, 1, True, 4), (64, 14, 256, 1024, 1, True, 4),   # weights resident: room for one a group
    (32, 150, 64, 128, 3, False, 4), (64, 56, 64, 64, 3, False, 8),
    (8, 28, 128, 512, 1, True, 0), (8, 56, 64, 256, 1, True, 0),       # few tiles a block
    (16, 56, 64, 256, 1, False, 0), (64, 56, 256, 256, 1, False, 0),   # no residual: the same, or operands need the memory
    (32, 75, 256, 256, 3, False, 0), (64, 56, 256, 32, 1, True, 0),    # long reductions, narrow tiles
], ids=str)
def test_layers_bound_by_their_rows_take_tile_buffers(N, HW, C, K, R, residual, buffers):
    d = q8.make_conv_desc(N, HW, HW, C, K, R, R, (1, 1), (R // 2, R // 2), relu=True)
    assert q8.q8_conv2d_query_row_buffers(d, None, residual) == buffers
    for y_type in (2, 3):   # 32-bit outputs are stored by the epilogue
        d.y_type = y_type
        assert q8.q8_conv2d_query_row_buffers(d, None, False) == 0


@pytest.mark.parametrize("N,HW,C,K,R,buffers", [(1, 112, 64, 256, 1, 8), (1, 56, 64, 128, 1, 0), (16, 56, 256, 512, 3, 2), (16, 56, 64, 64, 1, 0),
                                                (64, 56, 64, 64, 1, 8), (64, 56, 64, 32, 1, 0)], ids=str)
def test_residuals_of_fp32_outputs_come_through_tile_buffers(N, HW, C, K, R, buffers):
    d = q8.make_conv_desc(N, HW, HW, C, K, R, R, (1, 1), (R // 2, R // 2), y_type=q8.Q8_F32)
    assert q8.q8_conv2d_query_row_buffers(d, None, True) == buffers


@pytest.mark.parametrize("N,HW,C1,K1,K2,residual,buffers", [
    (64, 56, 64, 64, 256, True, 6), (64, 56, 64, 64, 256, False, 6), (4, 56, 64, 64, 256, True, 0),
    (64, 56, 128, 64, 256, True, 3), (32, 56, 64, 128, 512, True, 3),      # one a group, weights of the first layer resident
    (64, 56, 128, 128, 512, True, 3), (64, 28, 128, 128, 512, True, 0),    # streamed
    (64, 56, 128, 64, 256, False, 0), (64, 56, 64, 64, 128, False, 0),     # the first layer is most of the work
], ids=str)
def test_pairs_bound_by_their_rows_take_tile_buffers(N, HW, C1, K1, K2, residual, buffers):
    d1 = q8.make_conv_desc(N, HW, HW, C1, K1, 3, 3, (1, 1), (1, 1), relu=True)
    d2 = q8.make_conv_desc(N, HW, HW, K1, K2, 1, 1, relu=True)
    assert q8.q8_conv2d_query_row_buffers(d1, d2, residual) == buffers


def test_marshalled_calls_refuse_none_without_assertions():
    """In an interpreter that runs no assertions: an error of the argument, not an access to what it is not."""
    code = """if True:
        import torch, paper_1805_08691_b200 as q8
        from paper_1805_08691_b200 import binding
        for call in (lambda: binding._native.maxabs(None, None), lambda: binding._native.quantize(None, 1.0, q8.Q8_U8, None),
                     lambda: binding._native.dequantize(None, q8.Q8_U8, 1.0, None), lambda: q8.q8_calibrate_maxabs(None, None)):
            try:
                call()
            except AttributeError as e:
                if "numel" not in str(e):
                    raise
            else:
                raise SystemExit("no error")
        """
    assert subprocess.run([sys.executable, "-O", "-c", code], cwd=ROOT).returncode == 0


def test_marshalling_module_belongs_to_one_torch(monkeypatch):
    """Another torch asks for another file, which is built by a C++ compiler alone; without one the import says what is missing."""
    from paper_1805_08691_b200 import build
    import torch
    mine = build.native_path()
    assert os.path.exists(mine) and not build._native_stale()
    monkeypatch.setattr(torch, "__version__", "0.1+other")
    assert build.native_path() != mine and build._native_stale()
    monkeypatch.setattr(build.shutil, "which", lambda name: None)
    with pytest.raises(RuntimeError, match="compiler"):
        build.build_native()
    code = """if True:
        import torch
        torch.__version__ = "0.1+other"
        try:
            import paper_1805_08691_b200
        except ImportError as e:
            raise SystemExit(0 if "for this torch" in str(e) else 2)
        raise SystemExit("imported a module of another torch")
        """
    env = dict(os.environ, PATH="/nonexistent", CXX="/nonexistent")
    assert subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env).returncode == 0


@pytest.mark.parametrize("shape,operand", [((8, 99, 99, 3, 32, 3, 3), 3), ((8, 99, 99, 3, 64, 7, 1), 3), ((8, 99, 99, 3, 32, 1, 1), 3),
                                           ((8, 99, 99, 3, 32, 1, 7), 0), ((8, 99, 99, 4, 32, 3, 3), 0), ((8, 99, 99, 3, 24, 3, 3), 0),
                                           ((8, 99, 99, 3, 144, 3, 3), 0), ((1, 60, 60, 3, 32, 3, 3), 0)], ids=str)
def test_plan_tells_packed_operands_from_gathered_ones(shape, operand):
    plan = q8.q8_conv2d_query_plan(q8.make_conv_desc(*shape, x_type=q8.Q8_S8))
    assert plan.kernel == q8.Q8_KERNEL_GATHER and plan.operand == operand


@pytest.mark.parametrize("N,K,operand", [(10, 104, 0), (10, 52, 0), (1, 104, 0), (10, 48, 3), (10, 112, 3), (10, 44, 3)], ids=str)
@pytest.mark.parametrize("y_type", [2, 3])
def test_long_layers_with_ragged_32_bit_rows_are_gathered(y_type, N, K, operand):
    d = q8.make_conv_desc(N, 258, 258, 3, K, 3, 3, pad=(1, 1), y_type=y_type)
    assert q8.q8_conv2d_query_plan(d).operand == operand
    d.N, d.H = 1, 200   # 3.0 tiles a block
    assert q8.q8_conv2d_query_plan(d).operand == 3


def test_row_buffer_query_checks_what_it_is_given():
    d1 = q8.make_conv_desc(64, 56, 56, 64, 64, 3, 3, pad=(1, 1), relu=True)
    d2 = q8.make_conv_desc(64, 56, 56, 64, 256, 1, 1, relu=True)
    n = C.c_int(-1)
    assert q8.lib.q8_conv2d_query_row_buffers(C.byref(d1), None, 0, None) == 1
    assert q8.lib.q8_conv2d_query_row_buffers(None, None, 0, C.byref(n)) == 1 and n.value == -1
    bad = q8.make_conv_desc(64, 56, 56, 64, 0, 1, 1)
    assert _code(q8.q8_conv2d_query_row_buffers, bad) == 1 and _code(q8.q8_conv2d_query_row_buffers, d1, bad) == 1
    d1.K = d2.C = 256   # a pair that does not run as one launch
    assert q8.q8_conv2d_query_row_buffers(d1, d2, True) == 0
    d2.algo = q8.Q8_ALGO_DIRECT
    assert q8.q8_conv2d_query_row_buffers(d2, None, True) == 0
