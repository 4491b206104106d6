"""16-bit calls that need a channels-last copy, inside a stream capture: what may be done with the graph stays what it is for
calls that need none -- kernel nodes only, several executables, clones, a child of another graph, an update of an executable
-- and the copies' memory comes back when the graphs are gone."""
import pytest
import torch

pytestmark = pytest.mark.gpu
cr = pytest.importorskip("cuda.bindings.runtime")

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu


def _ok(ret):
    assert ret[0] == cr.cudaError_t.cudaSuccess, ret[0]
    return ret[1] if len(ret) == 2 else ret[1:]


def _capture(calls):
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        _ok(cr.cudaStreamBeginCapture(s.cuda_stream, cr.cudaStreamCaptureMode.cudaStreamCaptureModeGlobal))
        calls()
        return _ok(cr.cudaStreamEndCapture(s.cuda_stream))


def _instantiate(graph):
    return _ok(cr.cudaGraphInstantiate(graph, 0))


def _layer(Cin, Cout, ks):
    w = synth.kaiming_weights(24, Cin, Cout, Cin, ks)
    return gu.select_pack(w, ks, orc.pattern_preset(4, orc.PRESET_CENTRE8), 4, "bf16")[1]


def test_a_captured_call_leaves_the_graph_free():
    c, N, C, H, W = gu.ctx(), 2, 96, 40, 42
    packed = _layer(C, 80, 3)
    x = torch.randn((N, C, H, W), device="cuda").to(torch.bfloat16)
    y, want = (torch.zeros((N, 80, H, W), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    c.rtoss_conv3x3_pattern(packed, x, want, N, H, W)
    graph = _capture(lambda: [c.rtoss_conv3x3_pattern(packed, x, y, N, H, W) for _ in range(2)])
    n = _ok(cr.cudaGraphGetNodes(graph, 0))[1]
    nodes = _ok(cr.cudaGraphGetNodes(graph, n))[0]
    kinds = {_ok(cr.cudaGraphNodeGetType(v)) for v in nodes[:n]}
    assert n == 4 and kinds == {cr.cudaGraphNodeType.cudaGraphNodeTypeKernel}
    clone = _ok(cr.cudaGraphClone(graph))
    parent = _ok(cr.cudaGraphCreate(0))
    _ok(cr.cudaGraphAddChildGraphNode(parent, None, 0, graph))
    execs = [_instantiate(g) for g in (graph, graph, clone, parent)]
    again = _capture(lambda: [c.rtoss_conv3x3_pattern(packed, x, y, N, H, W) for _ in range(2)])
    _ok(cr.cudaGraphExecUpdate(execs[0], again))
    for g in (graph, clone, parent, again):     # (the executables hold the copies)
        _ok(cr.cudaGraphDestroy(g))
    s = torch.cuda.Stream()
    for e in execs:
        y.zero_()
        torch.cuda.synchronize()
        for _ in range(2):
            _ok(cr.cudaGraphLaunch(e, s.cuda_stream))
        torch.cuda.synchronize()
        assert torch.equal(y, want)
    for e in execs:
        _ok(cr.cudaGraphExecDestroy(e))
    assert c.rtoss_device_status() == 0
    packed.close()


def test_calls_of_a_capture_share_memory_only_in_order():
    """Calls one behind the other (growing, shrinking, a foreign kernel between them) and calls on a second stream of the same
    capture, which must not use the first one's copy while it is read: the results of calls one by one."""
    c, N = gu.ctx(), 4
    jobs = []
    for i, (C, H, W) in enumerate([(64, 60, 62), (96, 120, 90), (64, 60, 62), (80, 100, 90), (96, 120, 90), (64, 60, 62)]):
        packed = _layer(C, 72, 3)
        x = torch.randn((N, C, H, W), device="cuda").to(torch.bfloat16)
        y, want = (torch.zeros((N, 72, H, W), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        c.rtoss_conv3x3_pattern(packed, x, want, N, H, W)
        jobs.append((packed, x, y, want, H, W))
    other = torch.cuda.Stream()
    z = torch.zeros(1 << 20, device="cuda")

    def calls():
        here = torch.cuda.current_stream()
        for i, (packed, x, y, _, H, W) in enumerate(jobs):
            if i % 3 == 2:
                other.wait_stream(here)
                with torch.cuda.stream(other):
                    c.rtoss_conv3x3_pattern(packed, x, y, N, H, W)
            else:
                c.rtoss_conv3x3_pattern(packed, x, y, N, H, W)
                z.add_(1)
        here.wait_stream(other)

    e = _instantiate(_capture(calls))
    for _ in range(10):
        for j in jobs:
            j[2].zero_()
        torch.cuda.synchronize()
        _ok(cr.cudaGraphLaunch(e, torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        for j in jobs:
            assert torch.equal(j[2], j[3])
    _ok(cr.cudaGraphExecDestroy(e))
    assert c.rtoss_device_status() == 0
    for j in jobs:
        j[0].close()


def test_the_copies_come_back():
    c, N, C, H, W = rt.Context(0), 8, 64, 512, 512      # 256 MiB a copy
    packed = _layer(C, 16, 1)
    x = torch.zeros((N, C, H, W), dtype=torch.bfloat16, device="cuda")
    y = torch.empty((N, 16, H, W), dtype=torch.bfloat16, device="cuda")
    assert rt.rtoss_conv_route_of(N, H, W, 1, 1, rt.NCHW, rt.BF16, C, 16) == rt.ROUTE_TENSOR_REPACKED
    c.rtoss_conv1x1_pattern(packed, x, y, N, H, W)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for _ in range(12):
        graph = _capture(lambda: c.rtoss_conv1x1_pattern(packed, x, y, N, H, W))
        e = _instantiate(graph)
        _ok(cr.cudaGraphDestroy(graph))
        _ok(cr.cudaGraphLaunch(e, torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        _ok(cr.cudaGraphExecDestroy(e))
    assert free0 - torch.cuda.mem_get_info()[0] < 3 << 29       # (twelve copies are 3 GiB)
    graph = _capture(lambda: [c.rtoss_conv1x1_pattern(packed, x, y, N, H, W) for _ in range(12)])
    assert free0 - torch.cuda.mem_get_info()[0] < 3 << 29       # one behind the other: one copy
    _ok(cr.cudaGraphDestroy(graph))
    packed.close()
    c.close()
