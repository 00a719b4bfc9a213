"""GPU parity (bit-exact) of the tensor-core depthwise 3x3 kernel at the edges of its slabs, image groups and row runs."""
import numpy as np
import pytest
import torch

from paper_2202_05239_b200 import synth
from gpu_util import Guarded, api, assert_equal_arrays, random_conv_layer, random_input

pytestmark = pytest.mark.gpu

# (h, w, c, stride, n, x_signed, y_dtype)
CASES = [
    (14, 14, 512, 1, 33, False, synth.U8),      # four slabs, eight images a tile, the last group nearly empty
    (7, 7, 960, 1, 40, True, synth.S8),         # 15 slabs of 64 channels, 14 images a group
    (112, 112, 32, 1, 5, False, synth.U8),      # one slab of 32 channels, four images side by side, one in the last group
    (13, 17, 144, 1, 9, True, synth.U8),        # five slabs of 32, half of the last one empty, odd sizes
    (126, 126, 16, 1, 2, False, synth.S8),      # the widest row, 16 channels
    (1, 1, 128, 1, 300, False, synth.U8),       # a single position per image
    (3, 2, 96, 1, 7, True, synth.S8),
    (112, 112, 64, 2, 6, False, synth.U8),      # stride 2, even width
    (15, 13, 192, 2, 21, True, synth.S8),       # stride 2, odd sizes
    (7, 7, 1024, 2, 64, False, synth.U8),
    (2, 2, 48, 2, 3, True, synth.U8),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_depthwise(ref, request, case):
    h, w, c, stride, n, xs, y_dtype = CASES[case]
    rng = np.random.default_rng(4100 + case)
    a = api()
    layer = random_conv_layer(rng, h=h, w=w, c=c, c_out=c, k=3, stride=stride, pad=1, x_signed=xs, y_dtype=y_dtype, with_res=False,
                              kind=synth.DWCONV, fl_w=6, wide=bool(case & 1))
    x = random_input(rng, n, layer)
    want = ref.net_forward([layer], x)[-1]
    net = a.Net([layer], n)
    a.f8_debug_plan_options(32768)      # wherever the kernel applies, not only where it is the faster one
    request.addfinalizer(lambda: a.f8_debug_plan_options(0))
    before = a.f8_tc_launch_count()
    out = Guarded((n,) + net.out_shape, net.out_dtype)
    net.forward(a.to_device(x), out=out.t)
    torch.cuda.synchronize()
    a.f8_device_status()
    assert a.f8_tc_launch_count() == before + 1 and out.intact()
    assert_equal_arrays(out.t.cpu().numpy().reshape(want.shape), want, "output: ")
    net.close()


@pytest.mark.parametrize("h,c,stride,n,tensor_cores", [
    (56, 144, 1, 33, True),         # two images of 58 positions in a tile row
    (64, 144, 1, 33, False),        # one image of 66: half of every tile row is empty
    (78, 48, 1, 80, False),
    (98, 1232, 2, 1, False),        # one image in four blocks
    (112, 96, 2, 16, True),
    (7, 960, 1, 16, False),         # too few outputs to pay for the start
])
def test_which_kernel_a_depthwise_layer_takes(ref, h, c, stride, n, tensor_cores):
    rng = np.random.default_rng(h + c)
    a = api()
    layer = random_conv_layer(rng, h=h, w=h, c=c, c_out=c, k=3, stride=stride, pad=1, x_signed=False, y_dtype=synth.U8, with_res=False,
                              kind=synth.DWCONV, fl_w=6)
    x = random_input(rng, n, layer)
    net = a.Net([layer], n)
    before = a.f8_tc_launch_count()
    out = net.forward(a.to_device(x))
    torch.cuda.synchronize()
    a.f8_device_status()
    assert a.f8_tc_launch_count() - before == (1 if tensor_cores else 0)
    assert_equal_arrays(out.cpu().numpy().reshape(n, layer.ho, layer.wo, c), ref.run_layer(layer, x))
    net.close()
