"""A programmatic launch waits for the kernel before it and for nothing else:
in the graph that a training call leaves under stream capture, a node with a
programmatic edge in has no second edge in.  The graphs are inspected, never
launched."""

import ctypes

import pytest

from tests.gpu_common import lib_ready, torch_cuda

pytestmark = pytest.mark.gpu


class EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


PROGRAMMATIC = 1  # CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC


def captured_edges(torch, call):
    """[(source, target, programmatic)] of the graph of `call(stream)`."""
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(rc):
        assert rc == 0, rc

    stream = torch.cuda.Stream()
    st, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    torch.cuda.synchronize()
    ok(cu.cuStreamBeginCapture_v2(st, 0))
    try:
        with torch.cuda.stream(stream):
            call(stream)
    finally:
        rc = cu.cuStreamEndCapture(st, ctypes.byref(graph))
    ok(rc)
    ok(cu.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)))
    src, dst, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (EdgeData * n.value)()
    ok(cu.cuGraphGetEdges_v2(graph, src, dst, data, ctypes.byref(n)))
    ok(cu.cuGraphDestroy(graph))
    return [(src[i], dst[i], data[i].type == PROGRAMMATIC) for i in range(n.value)]


def check(edges):
    into = {}
    for _, b, _ in edges:
        into[b] = into.get(b, 0) + 1
    dependent = [b for _, b, p in edges if p]
    assert dependent  # inside a layer's chain the launches stay programmatic
    assert any(c > 1 for c in into.values())  # and the call does join streams
    assert [into[b] for b in dependent if into[b] > 1] == []


def pairs(torch, B, features):
    g = torch.Generator("cuda").manual_seed(B)
    x = torch.rand(2 * B, features, device="cuda", generator=g)
    y = torch.randint(0, 10, (2 * B,), device="cuda", dtype=torch.int32, generator=g)
    return x, y


@pytest.mark.parametrize("prec,images,fused", [("bf16", False, False), ("bf16", True, False), ("bf16", False, True),
                                               ("fp32", False, False)])
def test_net_steps(prec, images, fused):
    torch, ff = torch_cuda(), lib_ready()
    B, dims = 128, (784, 256, 264, 128)
    layers = [ff.Layer(dims[k], dims[k + 1], prec=prec, init_seed=k, max_rows=2 * B) for k in range(3)]
    for l in layers:
        l.set_fused_local_grad(fused)
    net = ff.Net(layers, max_B=B)
    x, y = pairs(torch, B, dims[0])

    def steps(stream):
        for _ in range(4):  # beyond the two batches a layer may run ahead
            if images:
                net.train_step_images(x[:B], y, stream=stream)
            else:
                net.train_step(x, y, B=B, stream=stream)
        net.sync(stream)

    steps(torch.cuda.current_stream())
    check(captured_edges(torch, steps))


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_performance_optimized_steps(prec):
    torch, ff = torch_cuda(), lib_ready()
    n, dims = 256, (784, 256, 264, 128)
    layers = [ff.Layer(dims[k], dims[k + 1], prec=prec, init_seed=k, max_rows=n) for k in range(3)]
    net = ff.PoNet(layers, [ff.Head(d, max_rows=n) for d in dims[1:]], max_rows=n)
    x, y = pairs(torch, n // 2, dims[0])

    def steps(stream):
        for _ in range(4):
            net.train_step(x, y, stream=stream)
        net.sync(stream)

    steps(torch.cuda.current_stream())
    check(captured_edges(torch, steps))


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_head_epoch_of_three_passes(prec):
    torch, ff = torch_cuda(), lib_ready()
    dims, B, n = (32, 64, 72), 2048, 2 * 16384 + 100
    layers = [ff.Layer(dims[k], dims[k + 1], prec=prec, init_seed=k) for k in range(2)]
    head = ff.Head(ff.Head.features_of(layers), max_rows=B)
    x, y = pairs(torch, n // 2, dims[0])

    def epoch(stream):
        head.train_epoch(layers, x, y, B, stream=stream)

    epoch(torch.cuda.current_stream())
    check(captured_edges(torch, epoch))


@pytest.mark.parametrize("mode,nodes", [("single_layer", 1), ("all_layers", 2)])
def test_chapter_schedule(mode, nodes):
    torch, ff = torch_cuda(), lib_ready()
    dims, P, B = (784, 256, 264, 128), 300, 128
    layers = [ff.Layer(dims[k], dims[k + 1], prec="bf16", init_seed=k) for k in range(3)]
    pff = ff.Pff(layers, P, B, 1, 3, mode=mode, nodes=nodes)
    x, _ = pairs(torch, P, dims[0])
    labels = torch.randint(0, 10, (3, 2 * P), device="cuda", dtype=torch.int32)
    check(captured_edges(torch, lambda stream: pff.run(x, labels, 0, 3, stream=stream)))
