"""Calls from several host threads."""
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
