"""Calls that are captured into a CUDA graph with no earlier call of their shape: whatever layout the handle has on the device by then
serves them, and the launch chosen for want of a better layout is not kept for later calls."""
import pytest
import torch

import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


def _layers(dtype, cin, cout, k, stride):
    """The same layer twice: one handle shows what to expect, the other has seen no call."""
    spec = synth.ConvSpec("c", cin, cout, k, stride, tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 15, cin + cout, 4, 4, "bernoulli", 0.4)
    return [nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, dtype) for _ in range(2)]


def _captured(lay, x):
    y = lay.alloc_out(x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lay(x, y)
    plan = rt3d.rt3d_last_plan()
    graph.replay()
    assert rt3d.rt3d_last_device_status() == rt3d.OK
    return y, plan


@pytest.mark.parametrize("prepared", [True, False])
def test_fp32_call_on_a_handle_without_a_call_of_its_shape(prepared):
    warm, lay = _layers(torch.float32, 64, 128, (3, 3, 3), (1, 1, 1))
    x = nets.to_device(synth.make_input(15, (2, 8, 28, 28, 64)), torch.float32)
    small = nets.to_device(synth.make_input(15, (1, 1, 4, 4, 64)), torch.float32)
    want, simt = warm(x), warm(x, algo=rt3d.ALGO_SIMT)
    warm(x)
    assert rt3d.rt3d_last_plan()["kernel"] == 8
    if prepared:
        lay.packed.prepare()
    else:                                                  # only the CUDA cores' layout is there
        lay(small)
        assert rt3d.rt3d_last_plan()["kernel"] == 0
    got, plan = _captured(lay, x)
    assert plan["kernel"] == (8 if prepared else 0)
    assert torch.equal(got, want) if prepared else float((got - simt).abs().max()) <= 2e-6 * float(simt.abs().max())
    assert torch.equal(lay(x), want) and rt3d.rt3d_last_plan()["kernel"] == 8


def test_narrow_layer_after_prepare():
    warm, lay = _layers(torch.bfloat16, 24, 64, (1, 3, 3), (1, 2, 2))
    x = nets.to_device(synth.make_input(15, (8, 8, 56, 56, 24)), torch.bfloat16)
    want = warm(x)
    plan = rt3d.rt3d_last_plan()
    assert plan["kernel"] == 2 and plan["tail_workers"] == 0
    lay.packed.prepare()                                   # steps of 64 channels
    got, captured = _captured(lay, x)
    assert captured == plan
    assert float((got - want).abs().max()) <= 2 ** -7 * float(want.abs().max())       # the same products in the same order
    assert torch.equal(lay(x), want)
