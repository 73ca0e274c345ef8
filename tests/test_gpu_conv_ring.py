"""The tensor-memory convolution with resident planes on other numbers of blocks than this chip's 152: a block's
first run of planes may then be shorter than one tile per issuing warp, and an issuer's first tile lie beyond the
ring's first fill (most numbers that are no multiple of four, 48 -> 16 and 32 -> 32 channels)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


class TcConvArgs(ctypes.Structure):
    _fields_ = [("s0", ctypes.c_void_p), ("s1", ctypes.c_void_p), ("c0", ctypes.c_int), ("c1", ctypes.c_int),
                ("m0", ctypes.c_int), ("m1", ctypes.c_int), ("No", ctypes.c_int), ("W", ctypes.c_void_p),
                ("bias", ctypes.c_void_p), ("out", ctypes.c_void_p), ("out32", ctypes.c_void_p),
                ("relu", ctypes.c_int), ("err", ctypes.c_void_p)]


@pytest.mark.parametrize("c0,up0,c1,cout", [(16, 0, 0, 16), (32, 1, 16, 16), (32, 0, 0, 32)])
def test_any_number_of_blocks(c0, up0, c1, cout):
    """The same bits on every number of blocks (each output is summed in one order), and within one BF16 rounding
    and K = 27 Cin FP32 roundings of the sum of magnitudes of the FP32 convolution."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1404_0959_gb300 import build
    lib = ctypes.CDLL(build.build())
    conv = getattr(lib, "_ZN2fe7conv_tcERKNS_10TcConvArgsEiiP11CUstream_st")
    N, cin = 128, c0 + c1
    g = torch.Generator(device="cuda").manual_seed(1)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    n0 = N // 2 if up0 else N
    a0 = rand(n0, n0, n0, c0).bfloat16()
    a1 = rand(N, N, N, c1).bfloat16() if c1 else None
    W, bias = (0.1 * rand(27, cout, cin)).bfloat16(), rand(cout)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")

    def run(blocks):
        out = torch.full((N, N, N, cout), float("nan"), device="cuda", dtype=torch.bfloat16)
        a = TcConvArgs(a0.data_ptr(), a1.data_ptr() if c1 else None, c0, c1, up0, 0, N, W.data_ptr(), bias.data_ptr(),
                       out.data_ptr(), None, 0, err.data_ptr())
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert conv(ctypes.byref(a), cout, blocks, stream) == 1
        torch.cuda.synchronize()
        assert int(err) == 0
        return out

    ref = run(152)
    for blocks in (1, 37, 121, 142, 146, 150, 151, 153, 159):
        assert torch.equal(run(blocks), ref), blocks
    # the convolution in plain torch, channels first, taps (dz, dy, dx)
    x = a0.float().permute(3, 0, 1, 2)[None]
    if up0:
        x = x.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
    if c1:
        x = torch.cat([x, a1.float().permute(3, 0, 1, 2)[None]], 1)
    x = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1), mode="circular")
    w = W.float().permute(1, 2, 0).reshape(cout, cin, 3, 3, 3)
    tf32 = torch.backends.cudnn.allow_tf32
    torch.backends.cudnn.allow_tf32 = False
    try:
        y = torch.nn.functional.conv3d(x, w, bias)[0]
        mag = torch.nn.functional.conv3d(x.abs(), w.abs(), bias.abs())[0]
    finally:
        torch.backends.cudnn.allow_tf32 = tf32
    d = (ref.float().permute(3, 0, 1, 2) - y).abs()
    assert bool((d <= 2.0 ** -8 * y.abs() + 2 * 27 * cin * 2.0 ** -24 * mag).all())
