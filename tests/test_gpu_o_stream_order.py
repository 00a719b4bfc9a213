"""Order of calls in one stream: blocks of a call may start while the call before it still runs, and what that call writes
(weights, biases, activations, shortcuts, sums) must be read complete.  Chains of calls over the same buffers, no
synchronisation in between, every result against the oracle."""
import numpy as np
import pytest
import torch

from oracle import f8fold
from paper_2202_05239_b200 import synth
from gpu_util import api, assert_equal_arrays, random_conv_layer

pytestmark = pytest.mark.gpu

FL_X, FL_W, FL_Y, FA = 5, 7, 3, 12
PASSES = 3


def _codes(acc, s, lo, hi):
    return np.clip((acc.astype(np.int64) + (1 << (s - 1))) >> s, lo, hi)


# (h, c, c_out, k, n, elements in front of the activations in the requantised tensor, kernel)
CHAINS = [
    (16, 16, 16, 3, 1, 0, "small"),
    (16, 16, 16, 3, 1, 20_000_000, "small"),           # the last part of a long tensor
    (14, 64, 64, 1, 1, 3_000_000, "small"),
    (28, 128, 128, 3, 6, 0, "tcgen05"),
    (28, 128, 128, 3, 6, 20_000_000, "tcgen05"),
    (14, 256, 256, 3, 8, 5_000_000, "tcgen05"),        # CTA pairs
    (15, 64, 40, 3, 9, 5_000_000, "tcgen05"),          # direct stores
]


@pytest.mark.parametrize("fold_first", [True, False])
@pytest.mark.parametrize("case", range(len(CHAINS)))
def test_chain_of_calls(ref, case, fold_first):
    """Compile step, requantisation, convolution with their weights, input and shortcut, convolution to 32 bits, requantisation."""
    a = api()
    h, c, c_out, k, n, lead, kernel = CHAINS[case]
    rng = np.random.default_rng(3000 + case)
    layer = random_conv_layer(rng, h=h, w=h, c=c, c_out=c_out, k=k, stride=1, pad=k // 2, x_signed=False, y_dtype=synth.U8, with_res=True,
                              fl_x=FL_X, fl_w=FL_W, fl_y=FL_Y, fl_r=4)
    layer.r_dtype = synth.S8
    nx, nr, kk = n * h * h * c, n * h * h * c_out, k * k * c
    total = lead + (max(nx, nr) + 15) // 16 * 16
    eta = f8fold.eta_fix(FL_X, 4.0)
    d = a.FoldDesc(c_out, kk, FL_X, FL_W, FL_W, eta, eta)
    sets, wants = [], []
    for _ in range(PASSES):
        w = rng.normal(0, 0.15, (c_out, kk)).astype(np.float32)
        vec = [rng.uniform(0.5, 1.5, c_out).astype(np.float32) for _ in range(4)]
        tail = rng.integers(-(1 << 16), 1 << 17, total - lead).astype(np.int32)
        w_q, b_q, _, _ = f8fold.fold_quantize(w, *vec, eta, eta, FL_X, FL_W, FL_W)
        x = _codes(tail, FA - FL_X, 0, 255)[:nx].astype(np.uint8).reshape(n, h, h, c)
        res = _codes(tail, FA - 4, -127, 127)[:nr].astype(np.int8).reshape(n, h, h, c_out)
        layer.weight[:] = w_q.reshape(layer.weight.shape)
        layer.bias[:] = b_q
        y8 = ref.run_layer(layer, x, res)
        y32 = ref.conv2d(x, layer.weight, layer.bias, stride=1, pad=k // 2, fl_x=FL_X, fl_w=FL_W, fl_y=0, y_dtype=synth.S32)
        wants.append((y8, y32, _codes(y32, FL_X + FL_W - 2, 0, 255), _codes(y32, FL_X + FL_W - 4, -127, 127)))
        acc = torch.zeros(total, dtype=torch.int32, device="cuda")
        acc[lead:] = torch.from_numpy(tail)
        sets.append(([a.to_device(t) for t in [w] + vec], acc))
    w_q = torch.empty(layer.weight.shape, dtype=torch.int8, device="cuda")
    b_q = torch.empty(c_out, dtype=torch.int32, device="cuda")
    fl = torch.empty(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(a.f8_fold_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    q1 = torch.empty(total, dtype=torch.uint8, device="cuda")
    q2 = torch.empty(total, dtype=torch.int8, device="cuda")
    x, res = q1[lead:lead + nx].view(n, h, h, c), q2[lead:lead + nr].view(n, h, h, c_out)
    desc, desc32 = a.conv_desc(layer, n), a.conv_desc(layer, n)
    desc32.y_dtype = synth.S32
    shape = (n, h, h, c_out)
    outs = [(torch.zeros(shape, dtype=torch.uint8, device="cuda"), torch.zeros(shape, dtype=torch.int32, device="cuda"),
             torch.zeros(shape, dtype=torch.uint8, device="cuda"), torch.zeros(shape, dtype=torch.int8, device="cuda")) for _ in range(4 * PASSES)]
    torch.cuda.synchronize()
    for i, (y8, y32, y_u, y_s) in enumerate(outs):
        (w, *vec), acc = sets[i % PASSES]

        def fold():
            a.f8_fold_quantize_fixed(d, w, *vec, w_q, b_q, fl, ws)
        if fold_first:
            fold()
        a.f8_requantize_dual_fixed(acc, FA, q1, synth.U8, FL_X, q2, synth.S8, 4)
        if not fold_first:
            fold()
        a.f8_conv2d_fixed(desc, x, w_q, b_q, res, y8)
        a.f8_conv2d_fixed(desc32, x, w_q, b_q, None, y32)
        a.f8_requantize_dual_fixed(y32, FL_X + FL_W, y_u, synth.U8, 2, y_s, synth.S8, 4)
    plan = a.f8_debug_last_plan()
    torch.cuda.synchronize()
    a.f8_device_status()
    assert bool(plan["m_tiles"]) == (kernel == "tcgen05")
    for i, got in enumerate(outs):
        for j, (g, want) in enumerate(zip(got, wants[i % PASSES])):
            assert_equal_arrays(g.cpu().numpy(), want, f"pass {i}, output {j}: ")


def test_compile_steps_that_share_a_workspace():
    """Two blocks' compile steps one behind the other through one workspace, over and over."""
    a = api()
    rng = np.random.default_rng(3100)
    eta_in, eta_out = f8fold.eta_fix(5, 4.0), f8fold.eta_fix(4, 6.0)
    steps = []
    for c_out, k, sigma in ((512, 4608, 0.02), (64, 147, 0.5), (2048, 512, 0.1), (17, 5, 2.0)):
        w = rng.normal(0, sigma, (c_out, k)).astype(np.float32)
        vec = [rng.uniform(0.5, 1.5, c_out).astype(np.float32) for _ in range(4)]
        want_w, want_b, want_fl, _ = f8fold.fold_quantize(w, *vec, eta_in, eta_out, 5, 0, 24)
        outs = [(torch.zeros((c_out, k), dtype=torch.int8, device="cuda"), torch.zeros(c_out, dtype=torch.int32, device="cuda"),
                 torch.zeros(1, dtype=torch.int32, device="cuda")) for _ in range(3)]
        steps.append((a.FoldDesc(c_out, k, 5, 0, 24, eta_in, eta_out), [a.to_device(t) for t in [w] + vec], outs, (want_w, want_b, want_fl)))
    ws = torch.empty(max(a.f8_fold_workspace_bytes(s[0]) for s in steps), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for rep in range(3):
        for d, dev, outs, _ in steps:
            a.f8_fold_quantize_fixed(d, *dev, *outs[rep], ws)
    torch.cuda.synchronize()
    for _, _, outs, (want_w, want_b, want_fl) in steps:
        for w_q, b_q, fl in outs:
            assert int(fl.item()) == want_fl
            assert_equal_arrays(w_q.cpu().numpy(), want_w)
            assert_equal_arrays(b_q.cpu().numpy(), want_b)
