"""Calls from several host threads."""
import sys
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from oracle import rtoss_oracle as orc
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu


def test_first_cuda_call_of_a_thread():
    """A thread whose first call to CUDA is a convolution that needs a tensor map (nothing has made a context current in it)."""
    c, masks = gu.ctx(), orc.pattern_preset(4, orc.PRESET_CENTRE8)
    _, packed = gu.select_pack(synth.kaiming_weights(23, 0, 96, 64, 3), 3, masks, 4, "bf16")
    x = torch.randn((2, 31, 33, 64), device="cuda").to(torch.bfloat16)
    y = torch.zeros((2, 2, 31, 33, 96), dtype=torch.bfloat16, device="cuda")
    c.rtoss_conv3x3_pattern(packed, x[:1], y[0], 1, 31, 33, 1, rt.NHWC)      # (what a device needs once is done here)
    torch.cuda.synchronize()
    stream, failed = torch.cuda.current_stream().cuda_stream, []
    desc = c._desc((2, 0, 31, 33), 1, rt.NHWC, rt.BF16, rt.ACT_NONE, None, 0, 0)

    def work():
        st = rt.lib.rtoss_conv3x3_pattern(c.h, packed.h, x.data_ptr(), y[1].data_ptr(), desc, stream)
        if st:
            failed.append(rt.lib.rtoss_last_error(c.h))

    t = threading.Thread(target=work)
    t.start()
    t.join()
    c.rtoss_conv3x3_pattern(packed, x, y[0], 2, 31, 33, 1, rt.NHWC)
    torch.cuda.synchronize()
    assert not failed and torch.equal(y[0], y[1])
    packed.close()


@pytest.mark.parametrize("ks,Cin", [(3, 64), (1, 72), (3, 50)])
def test_threads_share_a_context_and_a_handle(ks, Cin):
    """Four threads, each on a stream of its own, with more shapes than the context keeps tensor maps for, in the default layout
    and channels last: every result is the one a single thread gets, bit for bit (a call's order of sums depends on its sizes)."""
    c, Cout, masks = gu.ctx(), 80, orc.pattern_preset(4, orc.PRESET_CENTRE8)
    _, packed = gu.select_pack(synth.kaiming_weights(22, Cin, Cout, Cin, ks), ks, masks, 4, "bf16")
    fn = c.rtoss_conv3x3_pattern if ks == 3 else c.rtoss_conv1x1_pattern
    g = torch.Generator(device="cuda").manual_seed(3)
    jobs = []
    for i in range(48):      # (a context keeps 32 maps)
        H, W, layout = 40 + i % 7, 41 + i, rt.NCHW if i % 3 else rt.NHWC
        x = torch.empty((2, Cin, H, W) if layout == rt.NCHW else (2, H, W, Cin), device="cuda").normal_(generator=g).to(torch.bfloat16)
        y = [torch.zeros((2, Cout, H, W) if layout == rt.NCHW else (2, H, W, Cout), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        fn(packed, x, y[0], 2, H, W, 1, layout, rt.ACT_RELU)
        jobs.append((x, y, H, W, layout))
    torch.cuda.synchronize()
    failed, start = [], threading.Barrier(4)

    def work(t):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(5):
                    for x, y, H, W, layout in jobs[t::4]:
                        fn(packed, x, y[1], 2, H, W, 1, layout, rt.ACT_RELU)
        except Exception as e:   # (a thread's exception would be lost)
            failed.append(e)

    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-5)
    try:
        threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
        [t.start() for t in threads]
        [t.join() for t in threads]
    finally:
        sys.setswitchinterval(interval)
    torch.cuda.synchronize()
    assert not failed and c.rtoss_device_status() == 0
    for x, y, H, W, layout in jobs:
        assert torch.equal(y[0], y[1]), (H, W, layout)
    packed.close()
