"""GPU parity (bit-exact) of the kernel for layers of a few microseconds (mma.sync implicit GEMM), which f8_net_forward
takes for small dense layers: networks of one or two layers at the edges of its tiles and of its K chunks."""
import numpy as np
import pytest
import torch

from paper_2202_05239_b200 import synth
from gpu_util import Guarded, api, assert_equal_arrays, check_layer, random_conv_layer, random_input

pytestmark = pytest.mark.gpu

# (h, w, c, c_out, k, stride, pad, n, x_signed, y_dtype, with_res)
CASES = [
    (1, 1, 2048, 1000, 1, 1, 0, 1, False, synth.S32, False),     # a fully connected layer for one image
    (1, 1, 48, 16, 1, 1, 0, 33, True, synth.U8, False),          # 33 rows: one row in the second tile; K of 48 bytes
    (14, 14, 256, 256, 3, 1, 1, 1, False, synth.U8, True),       # 18 chunks through the eight-stage ring; shortcut
    (7, 9, 16, 48, 3, 2, 1, 3, True, synth.S8, False),           # one unit per tap: a chunk spans eight taps; ragged columns
    (15, 17, 80, 112, 5, 1, 2, 1, False, synth.U8, False),       # chunks straddle taps (80 of 128 bytes)
    (31, 29, 32, 64, 1, 2, 0, 2, False, synth.S8, False),        # strided 1x1
    (56, 56, 64, 256, 1, 1, 0, 1, False, synth.U8, True),        # 64 x 64 tiles
    (40, 41, 96, 272, 1, 1, 0, 2, True, synth.S8, True),         # 64 x 64 tiles, ragged in both directions
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_small_layer(ref, case):
    h, w, c, c_out, k, stride, pad, n, xs, y_dtype, with_res = CASES[case]
    rng = np.random.default_rng(2100 + case)
    layer = random_conv_layer(rng, h=h, w=w, c=c, c_out=c_out, k=k, stride=stride, pad=pad, x_signed=xs, y_dtype=y_dtype, with_res=with_res)
    layers = [layer]
    if with_res:      # the shortcut comes from a second layer over the same image
        short = random_conv_layer(rng, h=h, w=w, c=c, c_out=c_out, k=k, stride=stride, pad=pad, x_signed=xs, y_dtype=layer.r_dtype,
                                  with_res=False, fl_x=layer.fl_x)
        short.fl_y = layer.fl_r
        layer.res = 1
        layers = [short, layer]
    a = api()
    x = random_input(rng, n, layers[0])
    want = ref.net_forward(layers, x)
    net = a.Net(layers, n)
    guards = [Guarded((n, l.ho, l.wo, l.c_out), a.torch_dtype(l.y_dtype)) for l in layers]
    before = a.f8_tc_launch_count()
    net.forward(a.to_device(x), dump=[g.t for g in guards])
    torch.cuda.synchronize()
    a.f8_device_status()
    assert a.f8_tc_launch_count() - before == len(layers)
    for i, g in enumerate(guards):
        assert g.intact()
        assert_equal_arrays(g.t.cpu().numpy().reshape(want[i + 1].shape), want[i + 1], f"layer {i}: ")
    net.close()


def test_the_last_plan_is_not_that_of_an_earlier_call(ref):
    """f8_debug_last_plan reports the tcgen05 plan of the last call, and none where that call made none."""
    a = api()
    rng = np.random.default_rng(2300)
    large = random_conv_layer(rng, h=28, w=28, c=128, c_out=128, k=3, stride=1, pad=1, x_signed=False, y_dtype=synth.U8, with_res=False)
    small = random_conv_layer(rng, h=16, w=16, c=16, c_out=16, k=3, stride=1, pad=1, x_signed=False, y_dtype=synth.U8, with_res=False)
    xl, xs = a.to_device(random_input(rng, 2, large)), a.to_device(random_input(rng, 1, small))
    a.run_layer(large, xl)
    assert a.f8_debug_last_plan()["m_tiles"] > 0
    a.run_layer(small, xs)
    assert not any(a.f8_debug_last_plan().values())
    a.run_layer(large, xl)
    net = a.Net([small], 1)
    net.forward(xs)
    assert not any(a.f8_debug_last_plan().values())
    torch.cuda.synchronize()
    net.close()


# What a layer runs on by default: (h, w, c, c_out, k, stride, n, y_dtype, kernel in a network, kernel of a single-layer call)
ROUTES = [
    (16, 16, 16, 16, 3, 1, 1, synth.U8, "small", "small"),
    (14, 14, 256, 256, 3, 1, 1, synth.U8, "small", "tcgen05"),
    (31, 31, 16, 4096, 3, 1, 1, synth.U8, "tcgen05", "tcgen05"),      # more tiles than the machine holds at once
    (6, 6, 432, 96, 7, 2, 1, synth.S32, "tcgen05", "tcgen05"),        # two narrow tiles, 21168 products per output
    (13, 13, 48, 1784, 3, 1, 2, synth.U8, "small", "small"),          # rows of 1784 bytes, which the other kernel stores directly
    (17, 17, 768, 52, 3, 1, 7, synth.S32, "tcgen05", "tcgen05"),
    (20, 20, 1344, 184, 3, 1, 1, synth.S8, "tcgen05", "tcgen05"),
    (1, 1, 384, 128, 7, 1, 1, synth.U8, "cuda cores", "cuda cores"),  # one tap of 49 inside the image
    (1, 1, 2048, 1000, 1, 1, 1, synth.S32, "small", "cuda cores"),
    (1, 1, 4096, 1000, 1, 1, 1, synth.S32, "small", "small"),
]


@pytest.mark.parametrize("case", range(len(ROUTES)))
def test_which_kernel_a_layer_takes(ref, case):
    h, w, c, c_out, k, stride, n, y_dtype, in_net, alone = ROUTES[case]
    rng = np.random.default_rng(2400 + case)
    layer = random_conv_layer(rng, h=h, w=w, c=c, c_out=c_out, k=k, stride=stride, pad=k // 2, x_signed=False, y_dtype=y_dtype, with_res=False)
    a = api()

    def taken(before):
        tc = a.f8_tc_launch_count() - before
        return "tcgen05" if a.f8_debug_last_plan()["m_tiles"] else ("small" if tc else "cuda cores")
    x = random_input(rng, n, layer)
    before = a.f8_tc_launch_count()
    check_layer(ref, layer, x)
    assert taken(before) == alone
    net = a.Net([layer], n)
    before = a.f8_tc_launch_count()
    out = net.forward(a.to_device(x))
    assert taken(before) == in_net
    torch.cuda.synchronize()
    assert_equal_arrays(out.cpu().numpy().reshape(n, layer.ho, layer.wo, c_out), ref.run_layer(layer, x))
    net.close()


def test_current_stream_without_the_raw_handle(ref, monkeypatch):
    """The binding takes the current stream's handle straight from torch where it can; the Stream object gives the same one."""
    a = api()
    rng = np.random.default_rng(2500)
    layer = random_conv_layer(rng, h=12, w=12, c=32, c_out=32, k=3, stride=1, pad=1, x_signed=False, y_dtype=synth.U8, with_res=False)
    x = random_input(rng, 2, layer)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        handle = a._stream(None)
        assert handle == side.cuda_stream
        monkeypatch.setattr(a, "_raw_stream", None)
        assert a._stream(None) == handle
        out = a.run_layer(layer, a.to_device(x))
    assert a._stream(side) == handle
    side.synchronize()
    assert_equal_arrays(out.cpu().numpy(), ref.run_layer(layer, x))


# (h, w, c, c_out, k, stride, pad, n, x_signed, y_dtype, with_res): edges of the windows and of the panels
WINDOWS = [
    (2, 2, 1008, 32, 5, 1, 2, 1, False, synth.U8, False),       # weights of 25200 bytes a channel: several panels, the last one shorter
    (3, 5, 16, 16, 3, 1, 1, 7, False, synth.U8, True),          # one unit per tap, windows that cross images
    (9, 9, 48, 24, 3, 2, 1, 5, True, synth.S8, False),          # three units per tap, stride 2, columns past the last channel
    (13, 13, 112, 36, 3, 1, 1, 2, False, synth.S32, False),     # seven units per tap; an odd number of them in all
    (6, 11, 64, 260, 1, 2, 0, 3, False, synth.U8, False),       # skipped pixels
    (1, 7, 32, 20, 1, 1, 0, 2, True, synth.U8, True),           # fewer pixels than rows of a tile
    (12, 12, 32, 64, 3, 1, 0, 2, False, synth.U8, False),       # no padding: rows between two images that no filter starts at
    (11, 11, 64, 64, 2, 2, 0, 3, False, synth.U8, False),       # ... and that no filter reaches
    (8, 8, 128, 128, 7, 1, 3, 1, False, synth.U8, False),       # 49 taps
    # padding as large as the filter and larger: outputs, and whole rows of them, that read nothing but padding
    (8, 8, 32, 32, 3, 1, 3, 1, False, synth.U8, True),
    (12, 12, 64, 64, 1, 1, 1, 2, True, synth.S8, False),
    (9, 9, 16, 24, 2, 2, 2, 3, False, synth.U8, False),
    (5, 6, 48, 20, 1, 3, 2, 2, False, synth.S32, False),
    (7, 7, 32, 48, 3, 2, 5, 4, True, synth.U8, False),
    (1, 1, 2048, 64, 1, 1, 1, 1, False, synth.U8, False),
    (4, 4, 64, 72, 5, 1, 7, 2, False, synth.U8, False),
    # filters so large that only one of the smallest panels fits: two and three of them
    (11, 11, 32, 64, 25, 1, 12, 1, False, synth.U8, False),
    (8, 8, 32, 40, 29, 1, 14, 1, True, synth.U8, False),
    (9, 9, 48, 16, 25, 1, 12, 1, False, synth.S8, True),
]


@pytest.mark.parametrize("case", range(len(WINDOWS)))
def test_windows_and_panels(ref, case):
    h, w, c, c_out, k, stride, pad, n, xs, y_dtype, with_res = WINDOWS[case]
    rng = np.random.default_rng(2600 + case)
    layer = random_conv_layer(rng, h=h, w=w, c=c, c_out=c_out, k=k, stride=stride, pad=pad, x_signed=xs, y_dtype=y_dtype, with_res=with_res)
    layers = [layer]
    if with_res:
        short = random_conv_layer(rng, h=h, w=w, c=c, c_out=c_out, k=k, stride=stride, pad=pad, x_signed=xs, y_dtype=layer.r_dtype,
                                  with_res=False, fl_x=layer.fl_x)
        short.fl_y = layer.fl_r
        layer.res = 1
        layers = [short, layer]
    a = api()
    x = random_input(rng, n, layers[0])
    want = ref.net_forward(layers, x)
    net = a.Net(layers, n)
    out = Guarded((n, layer.ho, layer.wo, c_out), a.torch_dtype(y_dtype))
    before = a.f8_tc_launch_count()
    net.forward(a.to_device(x), out=out.t)
    torch.cuda.synchronize()
    a.f8_device_status()
    assert a.f8_tc_launch_count() - before == len(layers) and not a.f8_debug_last_plan()["m_tiles"], "another kernel took the layer"
    assert out.intact()
    assert_equal_arrays(out.t.cpu().numpy().reshape(want[-1].shape), want[-1])
    net.close()
