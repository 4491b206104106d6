"""Which kernels a call runs on (rtoss_conv_route_of, host arithmetic): one call of every kind, and the refusals."""
import pytest

from paper_2303_02191_b200 import binding as rt

F32, BF16, F16 = rt.F32, rt.BF16, rt.F16
CALLS = [
    # N, H, W, stride, ksize, layout, io type, Cin, Cout, path, handle's type -> route
    ((8, 80, 80, 1, 3, rt.NHWC, BF16, 128, 128, rt.PATH_AUTO, BF16), rt.ROUTE_TENSOR),
    ((8, 80, 80, 1, 3, rt.NHWC, F32, 128, 128, rt.PATH_AUTO, F32), rt.ROUTE_TENSOR),
    ((8, 80, 80, 1, 3, rt.NCHW, BF16, 128, 128, rt.PATH_AUTO, BF16), rt.ROUTE_TENSOR_REPACKED),
    ((3, 67, 101, 1, 3, rt.NHWC, F16, 100, 75, rt.PATH_AUTO, F16), rt.ROUTE_TENSOR_REPACKED),
    ((1, 640, 640, 2, 3, rt.NHWC, BF16, 3, 32, rt.PATH_AUTO, BF16), rt.ROUTE_STEM),
    ((1, 32, 32, 1, 3, rt.NCHW, F32, 32, 32, rt.PATH_AUTO, F32), rt.ROUTE_FEW),
    ((1, 32, 32, 1, 3, rt.NHWC, BF16, 32, 32, rt.PATH_FMA, BF16), rt.ROUTE_FEW),
    ((8, 80, 80, 1, 3, rt.NHWC, BF16, 128, 128, rt.PATH_FMA, BF16), rt.ROUTE_STAGED),
    ((8, 80, 80, 1, 3, rt.NHWC, BF16, 128, 128, rt.PATH_AUTO, F32), rt.ROUTE_STAGED),     # (the handle's type is not the data's)
    ((100, 1024, 1024, 1, 3, rt.NHWC, BF16, 150, 8, rt.PATH_AUTO, BF16), rt.ROUTE_TENSOR_REPACKED),
    ((200, 1024, 1024, 1, 3, rt.NHWC, BF16, 150, 8, rt.PATH_AUTO, BF16), rt.ROUTE_STAGED),   # (a copy of more than 2^31 pieces of 16 bytes)
    ((200, 1024, 1024, 1, 3, rt.NCHW, BF16, 150, 8, rt.PATH_AUTO, BF16), rt.ROUTE_STAGED),
    # where the few-outputs kernel was measured to be the slower one: one channel a warp, two a warp, pixels of whole vectors
    ((2, 31, 72, 1, 3, rt.NCHW, F16, 5, 215, rt.PATH_FMA, F16), rt.ROUTE_STAGED),
    ((2, 31, 72, 1, 3, rt.NCHW, F16, 17, 215, rt.PATH_FMA, F16), rt.ROUTE_FEW),
    ((1, 120, 100, 1, 3, rt.NHWC, F32, 13, 100, rt.PATH_FMA, F32), rt.ROUTE_STAGED),
    ((3, 23, 104, 1, 3, rt.NHWC, BF16, 96, 77, rt.PATH_FMA, BF16), rt.ROUTE_STAGED),
    ((3, 23, 104, 1, 3, rt.NHWC, BF16, 97, 77, rt.PATH_FMA, BF16), rt.ROUTE_FEW),
    ((14, 8, 28, 1, 3, rt.NCHW, F16, 6, 127, rt.PATH_AUTO, F16), rt.ROUTE_TENSOR_REPACKED),
    ((32, 80, 80, 1, 1, rt.NCHW, F32, 256, 256, rt.PATH_AUTO, F32), rt.ROUTE_STAGED),
]


@pytest.mark.parametrize("call,route", CALLS, ids=str)
def test_routes(call, route):
    assert rt.rtoss_conv_route_of(*call) == route


def test_refusals():
    for args, kw, status in (((1, 32, 32, 1, 3, rt.NCHW, BF16, 32, 32, rt.PATH_TENSOR), {}, rt.ERR_UNSUPPORTED),
                             ((1, 32, 32, 1, 3, rt.NCHW, BF16, 32, 32), dict(residual=True), rt.ERR_UNSUPPORTED),
                             ((1, 32, 32, 3, 3, rt.NCHW, BF16, 32, 32), {}, 1), ((1, 32, 32, 1, 5, rt.NCHW, BF16, 32, 32), {}, 1)):
        with pytest.raises(rt.RtossError) as e:
            rt.rtoss_conv_route_of(*args, **kw)
        assert e.value.status == status
