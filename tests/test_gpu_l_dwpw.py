"""GPU parity (bit-exact) of the kernel that runs a depthwise 3x3 layer and the pointwise layer behind it in one launch:
two- and three-layer networks at the edges of its slabs, parts and tiles, with and without a copy of the first output."""
import numpy as np
import pytest
import torch

from paper_2202_05239_b200 import synth
from gpu_util import Guarded, api, assert_equal_arrays, random_conv_layer, random_input

pytestmark = pytest.mark.gpu

# (h, w, c, c_out, stride, n, x_signed, y_dtype, with_res)
CASES = [
    (28, 28, 128, 64, 1, 3, False, synth.U8, False),       # one slab, one part
    (14, 14, 256, 256, 1, 9, True, synth.U8, False),       # two slabs, two parts, signed input
    (14, 14, 512, 512, 1, 3, False, synth.U8, False),      # four slabs stay staged under four parts, weights streamed
    (14, 14, 384, 64, 1, 5, False, synth.S8, False),       # three slabs through two slots
    (14, 14, 576, 160, 2, 4, False, synth.S8, False),      # stride 2, half a slab over, one part of 160 columns
    (13, 17, 144, 32, 1, 5, False, synth.S8, False),       # 16 channels in the second slab, 32-wide part, odd sizes
    (14, 14, 384, 384, 1, 150, False, synth.S8, True),     # shortcut, several tiles per CTA, three parts
    (7, 7, 960, 160, 1, 40, False, synth.S8, True),        # eight slabs, wide part, shortcut
    (56, 56, 64, 128, 2, 60, False, synth.U8, False),      # half a slab, many tiles per CTA
    (9, 7, 192, 96, 1, 130, True, synth.U8, True),         # ragged last tile, 96 of 128 columns, shortcut in u8 / s8
    # more slabs than slots and several tiles per CTA: the slots are used again while the epilogue of the tile before is open
    (14, 14, 384, 64, 1, 230, False, synth.S8, False),     # two accumulators, three or four tiles per CTA
    (14, 14, 320, 96, 1, 160, True, synth.S8, True),       # the same with a shortcut
    (37, 37, 400, 144, 1, 14, False, synth.U8, False),     # one wide part, one accumulator
    (13, 13, 544, 144, 1, 90, False, synth.U8, True),      # the same with five slabs and a shortcut
    (14, 14, 528, 160, 2, 420, True, synth.S8, False),     # the same at stride 2
]
SLOT_REUSE = {10: 2, 11: 2, 12: 1, 13: 1, 14: 1}           # case: accumulators of the pointwise layer


@pytest.mark.parametrize("case", range(len(CASES)))
def test_depthwise_pointwise(ref, request, case):
    h, w, c, c_out, stride, n, xs, y_dtype, with_res = CASES[case]
    rng = np.random.default_rng(3100 + case)
    a = api()
    dw = random_conv_layer(rng, h=h, w=w, c=c, c_out=c, k=3, stride=stride, pad=1, x_signed=xs, y_dtype=synth.U8, with_res=False,
                           kind=synth.DWCONV, fl_w=6)
    pw = random_conv_layer(rng, h=dw.ho, w=dw.wo, c=c, c_out=c_out, k=1, stride=1, pad=0, x_signed=False, y_dtype=y_dtype, with_res=with_res,
                           fl_x=dw.fl_y)
    layers = [dw, pw]
    pw.src = 1
    if with_res:
        short = random_conv_layer(rng, h=h, w=w, c=c, c_out=c_out, k=1, stride=1, pad=0, x_signed=xs, y_dtype=pw.r_dtype, with_res=False, fl_x=dw.fl_x)
        short.fl_y = pw.fl_r
        dw.src, pw.src, pw.res = 0, 2, 1
        layers = [short, dw, pw]
    x = random_input(rng, n, layers[0])
    want = ref.net_forward(layers, x)
    if case in SLOT_REUSE:
        lay = a.f8_debug_dwpw_layout(a.conv_desc(dw, n), c_out, with_res)
        assert lay["accs2"] == SLOT_REUSE[case] and lay["slabs"] > lay["slots"] and lay["tiles"] > 148 * lay["accs2"]
    net = a.Net(layers, n)
    a.f8_debug_plan_options(32768)      # the pair in one launch wherever the kernel applies, not only where it is the faster one
    request.addfinalizer(lambda: a.f8_debug_plan_options(0))
    xd = a.to_device(x)
    guards = [Guarded((n, l.ho, l.wo, l.c_out), a.torch_dtype(l.y_dtype)) for l in layers]
    for dump in (None, [g.t for g in guards]):
        out = Guarded((n,) + net.out_shape, net.out_dtype)
        ws = Guarded((net.workspace_bytes(n),), torch.uint8)
        net.forward(xd, out=out.t, workspace=ws.t, dump=dump)
        torch.cuda.synchronize()
        a.f8_device_status()
        assert net.fused_pairs == 1 and out.intact() and ws.intact()
        assert_equal_arrays(out.t.cpu().numpy().reshape(want[-1].shape), want[-1], f"output, dump {dump is not None}: ")
    for i, g in enumerate(guards):
        assert g.intact()
        assert_equal_arrays(g.t.cpu().numpy().reshape(want[i + 1].shape), want[i + 1], f"layer {i}: ")
    net.close()
