"""rtoss_packed_to_dense at the sizes where a block's share changes: fewer kernels than a block takes, one more, one block per SM
with a ragged last share, shares that fill a block's registers or its shared memory, several blocks an SM, and blocks that take
a second step.  Bit for
bit the weights under their masks, rounded to the handle's type."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2303_02191_b200 import binding as rt
    import gpu_util as gu

TD = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.mark.parametrize("cout,cin,ks,k,dt", [
    (1, 1, 3, 4, "bf16"), (16, 16, 3, 4, "bf16"), (257, 1, 3, 4, "f16"), (5, 13, 1, 3, "bf16"),
    (148, 256, 3, 4, "bf16"), (149, 257, 3, 2, "f16"),          # one block an SM, with and without a remainder
    (512, 331, 3, 4, "bf16"),                                    # more words a thread than it holds in registers
    (331, 331, 3, 9, "f32"),                                     # the same in fp32
    (700, 600, 3, 5, "f32"),                                     # as many kernels as fit, and more than one block an SM
    (1100, 1101, 3, 9, "f32"),                                   # 1008 kernels a step: 18 of eight blocks an SM take a second one
    (2, 3, 1, 4, "bf16"),                                        # nothing but trailing weights
    (2048, 1031, 1, 4, "bf16"),                                  # a 1x1 layer with trailing weights
])
def test_to_dense_is_the_masked_weights(cout, cin, ks, k, dt):
    c = gu.ctx()
    masks = rt.rtoss_pattern_preset(k, {4: rt.PRESET_CENTRE8, 9: rt.PRESET_DENSE}.get(k, rt.PRESET_CONN4))
    g = torch.Generator(device="cuda")
    g.manual_seed(cout + cin)
    w = torch.randn(cout, cin, ks, ks, device="cuda", generator=g)
    pid = c.rtoss_select_patterns(w, ks, masks, k)
    packed = c.rtoss_pack(w, ks, masks, k, pid, rt.DTYPE_NAMES[dt])
    out = torch.full((w.numel() + 8,), 7.0, dtype=TD[dt], device="cuda")
    c._check(rt.lib.rtoss_packed_to_dense(c.h, packed.h, out.data_ptr(), torch.cuda.current_stream().cuda_stream))
    table = torch.tensor([int(m) for m in masks], device="cuda")
    n = w.numel() // 9
    keep = (table[pid.reshape(-1)[:n].long()][:, None] >> torch.arange(9, device="cuda")) & 1
    want = torch.zeros(w.numel(), device="cuda")
    want[:9 * n] = torch.where(keep.reshape(-1) != 0, w.reshape(-1)[:9 * n], torch.zeros((), device="cuda"))
    assert torch.equal(out[:w.numel()], want.to(TD[dt]))
    assert torch.all(out[w.numel():] == 7.0)
    packed.close()


def test_a_refused_launch_is_reported_once():
    """The legacy stream takes no work while a stream that it waits for is captured: that call says so, and the next one, which is
    in order, is not answered with its error."""
    c = gu.ctx()
    masks = rt.rtoss_pattern_preset(4, rt.PRESET_CENTRE8)
    w = torch.randn(32, 16, 3, 3, device="cuda")
    pid = c.rtoss_select_patterns(w, 3, masks, 4)
    packed = c.rtoss_pack(w, 3, masks, 4, pid, rt.BF16)
    out = packed.to_dense()   # (what a first call sets up is done)
    torch.cuda.synchronize()
    cudart = ctypes.CDLL("libcudart.so.12")
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert cudart.cudaStreamCreate(ctypes.byref(stream)) == 0
    assert cudart.cudaStreamBeginCapture(stream, 0) == 0
    refused = rt.lib.rtoss_packed_to_dense(c.h, packed.h, out.data_ptr(), None)
    assert cudart.cudaStreamEndCapture(stream, ctypes.byref(graph)) != 0   # (the capture did not survive it)
    cudart.cudaGetLastError()
    cudart.cudaStreamDestroy(stream)
    assert refused != rt.OK
    assert torch.equal(pid, c.rtoss_select_patterns(w, 3, masks, 4))
    torch.cuda.synchronize()
    packed.close()
