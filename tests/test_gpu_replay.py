"""QuantNetwork.forward replays recorded launches: it must give what its layers launched one by one give, bit for bit, for
new images, on any stream, inside a caller's capture, and after any of the tensors, descriptors or factors that the
layers run with has been replaced."""
import copy
import pickle
import threading

import numpy as np
import pytest
import torch

from paper_1805_08691_b200 import network
from tests.test_oracle_network import _calibrate, _conv, _fold, _mini_inception
from workloads import nets
from workloads.nets import Layer
from workloads.synth import rng

pytestmark = pytest.mark.gpu

BATCH = 2


def _normalised_heads():
    """conv -> conv -> L2 normalisation -> two heads that run as one launch, and a residual block beside them."""
    g = rng(91)
    L = []
    x = _conv(g, L, "c1", "input", 3, 32, 3, pad=1)
    y = _conv(g, L, "c2", x, 32, 64, 3, pad=1)
    L.append(Layer("c2_norm", "l2norm", [y], gamma=np.full(64, 20.0, np.float32)))
    _conv(g, L, "head_a", "c2_norm", 64, 8, 3, pad=1, relu=False, bn=False, bias=True, f32_out=True)
    _conv(g, L, "head_b", "c2_norm", 64, 12, 3, pad=1, relu=False, bn=False, bias=True, f32_out=True)
    L.append(Layer("pool", "maxpool", [x], k=(2, 2), stride=(2, 2)))
    _conv(g, L, "c3", x, 32, 32, 1, residual=x)
    return L


LISTS = {"heads": (_normalised_heads, 24), "inception": (_mini_inception, 12),
         "bottlenecks": (lambda: nets.bottleneck_stack(C=64, blocks=2), 32)}


def _network(name, **kw):
    layers, hw = LISTS[name][0](), LISTS[name][1]
    folded = _fold(layers)
    maxima = _calibrate(layers, folded, 91, 1, hw)
    cuda = {n: tuple(None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in wb) for n, wb in folded.items()}
    return network.QuantNetwork(layers, cuda, maxima, (BATCH, hw, hw, 3), **kw)


def _images(name, seed):
    return torch.from_numpy(nets.images(seed, BATCH, LISTS[name][1])).cuda()


def _snapshot(out):
    torch.cuda.synchronize()
    return {k: v.clone() for k, v in out.items()}


def _poison(net):
    for b in net.bufs.values():
        b.fill_(3)


def _one_by_one(net, x):
    """The same forward with its layers enqueued by the host."""
    from paper_1805_08691_b200 import binding as q8
    _poison(net)
    q8.q8_quantize_pad_image(x, net.w_pad_in, net.c_pad_in, net.info["input"][1], q8.Q8_S8, out=net.bufs["input"])
    net._run_layers()
    return _snapshot(net.outputs)


def _assert_same(got, want):
    torch.cuda.synchronize()
    assert got.keys() == want.keys()
    for k in want:
        assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("streams", [1, 4])
@pytest.mark.parametrize("name", LISTS)
def test_new_images_other_streams_and_a_callers_capture(q8, name, streams):
    net = _network(name, streams=streams)
    for seed in (1, 2):
        x = _images(name, seed)
        want = _one_by_one(net, x)
        _poison(net)
        _assert_same(_snapshot(net.forward(x)), want)
        _poison(net)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            out = net.forward(x)
        side.synchronize()
        _assert_same(_snapshot(out), want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = net.forward(x)
    for seed in (3, 4):
        y = _images(name, seed)
        want = _one_by_one(net, y)
        x.copy_(y)
        _poison(net)
        graph.replay()
        _assert_same(_snapshot(out), want)
    q8.q8_read_status()


def _new_weights(net):
    net.convs["c2"].w_q = net.convs["c2"].w_q.flip(0).contiguous()


def _new_weight_storage(net):
    net.convs["c2"].w_q.data = net.convs["c2"].w_q.flip(0).contiguous()


def _weights_in_place(net):
    net.convs["c2"].w_q.copy_(net.convs["c2"].w_q.flip(0))


def _new_layer(net):
    import dataclasses
    qc = net.convs["c1"]
    net.convs["c1"] = dataclasses.replace(qc, b_q=qc.b_q + 100, scale=qc.scale * 0.5)


def _no_bias(net):
    net.convs["c2"].b_q = None


def _descriptor(net):
    net.convs["head_a"].desc.relu = 1


def _residual_factor(net):
    net.convs["c3"].res_scale *= 0.5


def _buffer(net):
    net.bufs["c1"] = torch.zeros_like(net.bufs["c1"])


def _normalisation(net):
    q, eps, mult = net.l2["c2_norm"]
    net.l2["c2_norm"] = (q, 100.0, mult * 0.5)


@pytest.mark.parametrize("change", [_new_weights, _new_weight_storage, _weights_in_place, _new_layer, _no_bias, _descriptor,
                                    _residual_factor, _buffer, _normalisation], ids=lambda f: f.__name__[1:])
def test_what_is_replaced_after_construction_takes_effect(q8, change):
    net = _network("heads", streams=2, fuse=False)
    x = _images("heads", 1)
    before = _snapshot(net.forward(x))
    change(net)
    _poison(net)
    net.forward(x)
    got = _snapshot(net.bufs)
    want = _one_by_one(net, x)
    _assert_same(got, _snapshot(net.bufs))
    if change is not _buffer:
        assert any(not torch.equal(before[k], want[k]) for k in want)
    q8.q8_read_status()


@pytest.mark.parametrize("layer", ["stem", "m0_3x1", "m1_3x3_s2"])
def test_a_layer_that_is_refused_raises_its_own_error(q8, layer):
    """... from the forward that would launch it, whichever stream it is on; the network works again once it is mended."""
    net = _network("inception", streams=4)
    x = _images("inception", 1)
    want = _one_by_one(net, x)
    stride = net.convs[layer].desc.stride_h
    net.convs[layer].desc.stride_h = 0
    for _ in range(2):
        with pytest.raises(q8.Q8Error) as e:
            net.forward(x)
        assert e.value.code == 1
    net.convs[layer].desc.stride_h = stride
    _poison(net)
    _assert_same(_snapshot(net.forward(x)), want)
    q8.q8_read_status()


def test_a_refused_layer_does_not_prevent_construction(q8, monkeypatch):
    def refuse(*a, **k):
        raise q8.Q8Error(2, "refused")
    with monkeypatch.context() as m:
        m.setattr(network.q8, "q8_maxpool2d", refuse)
        net = _network("inception", streams=4)
        x = _images("inception", 1)
        with pytest.raises(q8.Q8Error, match="refused"):
            net.forward(x)
    want = _one_by_one(net, x)
    _poison(net)
    _assert_same(_snapshot(net.forward(x)), want)


def test_recording_leaves_other_threads_alone(q8, monkeypatch):
    """While the launches of a network are recorded, another thread's work on any stream of the framework's pool runs (it is
    not recorded), and it may draw random numbers."""
    pool = [torch.cuda.Stream() for _ in range(32)]
    counts = [torch.zeros(1, device="cuda") for _ in pool]
    torch.cuda.synchronize()
    failed, rounds, launch = [], [], network.q8.q8_maxpool2d

    def work():
        try:
            for st, c in zip(pool, counts):
                with torch.cuda.stream(st):
                    c.add_(1)
            torch.rand(4, device="cuda")
        except Exception as e:
            failed.append(e)

    def maxpool(*a, **k):
        t = threading.Thread(target=work)
        t.start()
        t.join()
        rounds.append(1)
        return launch(*a, **k)

    with monkeypatch.context() as m:
        m.setattr(network.q8, "q8_maxpool2d", maxpool)
        net = _network("inception", streams=4)
    assert rounds and not failed
    for st, c in zip(pool, counts):
        st.synchronize()
        assert c.item() == len(rounds)
    x = _images("inception", 1)
    want = _one_by_one(net, x)
    _poison(net)
    _assert_same(_snapshot(net.forward(x)), want)
    assert [c.item() for c in counts] == [len(rounds)] * len(pool)


@pytest.mark.parametrize("duplicate", [copy.deepcopy, lambda net: pickle.loads(pickle.dumps(net))], ids=["deepcopy", "pickle"])
def test_a_copied_network_runs_on_its_own_tensors(q8, duplicate):
    net = _network("bottlenecks", streams=1)
    x, y = _images("bottlenecks", 1), _images("bottlenecks", 2)
    want_x, want_y = _one_by_one(net, x), _one_by_one(net, y)
    twin = duplicate(net)
    a, b = net.forward(x), twin.forward(y)
    _assert_same(_snapshot(a), want_x)
    _assert_same(_snapshot(b), want_y)
