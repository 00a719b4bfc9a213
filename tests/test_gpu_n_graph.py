"""GPU parity of repeated forward passes, which go out as one CUDA graph once a plan has been used often enough."""
import numpy as np
import pytest
import torch

from paper_2202_05239_b200 import synth
from gpu_util import api, assert_equal_arrays

pytestmark = pytest.mark.gpu

AFTER = 16         # passes of a plan before its launches are kept as a graph


@pytest.mark.parametrize("name,batch,image", [("resnet18", 3, 64), ("resnet50", 1, 96), ("mobilenetv2", 2, 64), ("resnet18_siblings", 2, 64)])
def test_repeated_passes(ref, name, batch, image):
    a = api()
    layers = synth.make_net(name, 0, image=image)
    hosts = [synth.draw_image(batch, s, image, image) for s in (1, 2)]
    wants = [ref.net_forward(layers, h, keep_all=False)[-1] for h in hosts]
    net = a.Net(layers, batch)
    x = a.to_device(hosts[0])
    out = torch.empty((batch,) + net.out_shape, dtype=net.out_dtype, device="cuda")
    ws = torch.empty(net.workspace_bytes(batch), dtype=torch.uint8, device="cuda")
    other = torch.empty_like(out)
    side = torch.cuda.Stream()
    counts = []

    def check(which, **kw):
        x.copy_(torch.from_numpy(hosts[which]))
        o = kw.pop("out", out)
        o.zero_()
        torch.cuda.synchronize()
        before = a.f8_tc_launch_count()
        net.forward(x, out=o, workspace=ws, **kw)
        torch.cuda.synchronize()
        a.f8_device_status()
        if "dump" not in kw:
            counts.append((net.last_launch_count, a.f8_tc_launch_count() - before))
        assert_equal_arrays(o.cpu().numpy(), wants[which])

    for i in range(AFTER + 3):               # the input changes in place
        check(i & 1)
        assert net.graph_info["last"] == (i >= AFTER)
    assert net.graph_info["made"] == 1
    check(1, stream=side)                    # on another stream
    assert net.graph_info == {"last": 1, "made": 1, "updates": 0, "failed": 0}
    check(0, out=other)                      # another output, then the first one: the same graph with other parameters
    last = net.graph_info["updates"]         # launches that read the input or write the output
    assert last > 0
    check(1)
    check(1, out=other)
    assert net.graph_info == {"last": 1, "made": 1, "updates": 3 * last, "failed": 0}
    first, x = x, torch.empty_like(x)        # ... and another input
    check(0)
    assert net.graph_info == {"last": 1, "made": 1, "updates": 4 * last, "failed": 0}
    check(1, out=other)
    x = first
    check(0)
    assert net.graph_info["last"] == 1 and net.graph_info["made"] == 1
    check(0, dump=[net.layer_output(i, batch) for i in range(len(layers))])
    assert net.graph_info["last"] == 0
    for i in range(AFTER + 1):               # another plan now
        check(i & 1)
    assert net.graph_info["last"] == 1 and net.graph_info["made"] == 2
    net.set_profiling(True)
    check(0)
    assert net.graph_info["last"] == 0
    net.set_profiling(False)
    for i in range(AFTER + 1):
        check(i & 1)
    assert net.graph_info["last"] == 1 and net.graph_info["made"] == 3
    try:                                     # kernels carry the bound of their waits: a new one means new launches
        a.f8_debug_set_wait_limit_ms(1500.0)
        check(1)
        assert net.graph_info["last"] == 0
        for i in range(AFTER):
            check(i & 1)
        assert net.graph_info["last"] == 1 and net.graph_info["made"] == 4
    finally:
        a.f8_debug_set_wait_limit_ms(0.0)
    for i in range(AFTER + 1):
        check(i & 1)
    assert net.graph_info["last"] == 1 and net.graph_info["failed"] == 0
    assert len(set(counts)) == 1
    # inside a caller's capture the launches become the caller's
    g = torch.cuda.CUDAGraph()
    check(1)
    with torch.cuda.graph(g, stream=side):
        net.forward(x, out=out, workspace=ws, stream=torch.cuda.current_stream())
        assert net.graph_info["last"] == 0
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert_equal_arrays(out.cpu().numpy(), wants[1])
    del g
    check(0)
    assert net.graph_info["last"] == 1
    net.close()


def test_batches_in_turns_make_no_graph(ref):
    """A plan that is left before its graph would pay costs what its launches cost."""
    a = api()
    layers = synth.make_net("resnet18", 0, image=64)
    host = synth.draw_image(3, 1, 64, 64)
    want = ref.net_forward(layers, host, keep_all=False)[-1]
    net = a.Net(layers, 3)
    x = a.to_device(host)
    ws = torch.empty(net.workspace_bytes(3), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        for n in (1, 3):
            for _ in range(AFTER):
                out = net.forward(x[:n], workspace=ws)
            torch.cuda.synchronize()
            assert_equal_arrays(out.cpu().numpy(), want[:n])
    assert net.graph_info["made"] == 0
    net.close()


def test_launch_count_behind_a_pass_of_no_images():
    a = api()
    layers = synth.make_net("resnet18", 0, image=64)
    net = a.Net(layers, 2)
    x = a.to_device(synth.draw_image(2, 1, 64, 64))
    out = torch.empty((2,) + net.out_shape, dtype=net.out_dtype, device="cuda")
    ws = torch.empty(net.workspace_bytes(2), dtype=torch.uint8, device="cuda")
    for _ in range(AFTER + 2):
        net.forward(x, out=out, workspace=ws)
    assert net.graph_info["last"] == 1
    launches = net.last_launch_count
    assert launches > 4
    net.forward(x[:0], out=out[:0], workspace=ws)
    assert net.last_launch_count == 0
    net.forward(x, out=out, workspace=ws)
    assert net.last_launch_count == launches
    torch.cuda.synchronize()
    net.close()


def test_last_plan_of_a_pass_with_other_buffers():
    """f8_debug_last_plan reports the pass's plan, also when only the steps at the caller's tensors were planned again."""
    a = api()
    layers = synth.make_net("resnet50", 0, image=96)
    net = a.Net(layers, 8)
    x = a.to_device(synth.draw_image(8, 1, 96, 96))
    ws = torch.empty(net.workspace_bytes(8), dtype=torch.uint8, device="cuda")
    outs = [torch.empty((8,) + net.out_shape, dtype=net.out_dtype, device="cuda") for _ in range(2)]
    net.forward(x, out=outs[0], workspace=ws)
    plan = a.f8_debug_last_plan()
    assert plan["m_tiles"] > 0
    net.forward(x, out=outs[1], workspace=ws)
    assert a.f8_debug_last_plan() == plan
    net.forward(x.clone(), out=outs[0], workspace=ws)
    assert a.f8_debug_last_plan() == plan
    torch.cuda.synchronize()
    net.close()


def test_a_graph_that_cannot_be_made_is_tried_again(ref):
    """The failure is made on the host.  The passes go out launch by launch meanwhile; another plan tries at once, the same one later."""
    a = api()
    layers = synth.make_net("resnet18", 0, image=64)
    host = synth.draw_image(2, 1, 64, 64)
    want = ref.net_forward(layers, host, keep_all=False)[-1]
    net = a.Net(layers, 2)
    x = a.to_device(host)
    out = torch.empty((2,) + net.out_shape, dtype=net.out_dtype, device="cuda")
    spaces = [torch.empty(net.workspace_bytes(2), dtype=torch.uint8, device="cuda") for _ in range(2)]

    def passes(n, ws):
        for _ in range(n):
            out.zero_()
            net.forward(x, out=out, workspace=ws)
        torch.cuda.synchronize()
        assert_equal_arrays(out.cpu().numpy(), want)
        return net.graph_info
    try:
        a.f8_debug_fail_graphs(2)
        assert passes(40, spaces[0]) == {"last": 0, "made": 0, "updates": 0, "failed": 1}
        info = passes(40, spaces[1])                     # another plan: its first attempt fails too
        assert (info["made"], info["failed"]) == (0, 2)
        info = passes(40, spaces[0])
        assert (info["last"], info["made"], info["failed"]) == (1, 1, 2)
        a.f8_debug_fail_graphs(1)
        info = passes(40, spaces[1])
        assert (info["last"], info["made"], info["failed"]) == (0, 1, 3)
        info = passes(100, spaces[1])                    # the same plan
        assert (info["last"], info["made"], info["failed"]) == (1, 2, 3)
    finally:
        a.f8_debug_fail_graphs(0)
    net.close()
