"""Repeated calls: a network's noted forward pass and a handle's prepared calls give the bits of first calls, and are
dropped when what they were made from changes."""
import pytest
import torch

import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets
import bench

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,clip", [("c3d", (16, 112, 112, 3)), ("r2plus1d", (4, 56, 56, 3)), ("s3d", (8, 96, 96, 3))])
def test_noted_forward_gives_the_bits_of_the_first(name, clip):
    net, _ = bench.build_network(name)
    xs = [nets.to_device(synth.make_input(9 + i, (2,) + clip)) for i in range(3)]
    first = [net._forward(x, 0, None, None).clone() for x in xs]
    for x, want in list(zip(xs, first)) * 2:                      # another input address each time
        assert torch.equal(net.forward(x), want)
    assert len(net._noted) == 1
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):                                 # another current stream
        got = net.forward(xs[1]).clone()
    side.synchronize()
    assert torch.equal(got, first[1])
    small = nets.to_device(synth.make_input(3, (1,) + clip))      # another shape in between
    want = net._forward(small, 0, None, None).clone()
    for _ in range(2):
        assert torch.equal(net.forward(small), want)
        assert torch.equal(net.forward(xs[2]), first[2])
    layer = next(iter(net.layers.values()))
    layer.bias = layer.bias + 1.0                                 # a changed layer must not run from the old notes
    changed = net.forward(xs[0]).clone()
    assert torch.equal(changed, net._forward(xs[0], 0, None, None)) and not torch.equal(changed, first[0])
    graph = nets.GraphedForward(net, xs[0])
    assert torch.equal(graph(), changed)
    assert rt3d.rt3d_last_device_status() == rt3d.OK


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_prepared_calls_of_a_handle(dtype):
    """More distinct calls than a handle remembers, in turn: every one keeps giving its own result, and a layer that
    replaces another at the same address is not taken for it."""
    spec = synth.ConvSpec("l", 64, 64, (3, 3, 3), (1, 1, 1), (1, 1, 1), True)
    L = synth.make_layer(spec, 3, 0, 4, 4, "bernoulli", 0.4)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, dtype)
    xs = [nets.to_device(
                  synth.make_input(i, (1, 2 + i % 3, 9, 8 + i, 64)), dtype) for i in range(11)]
    want = [lay(x).clone() for x in xs]
    ys = [torch.zeros_like(w) for w in want]
    for _ in range(3):
        for x, y, w in zip(xs, ys, want):
            y.zero_()
            lay(x, y)
            assert torch.equal(y, w)
            lay(x, y, relu=False)
            assert bool((y < 0).any())
    for seed in range(1, 5):
        L = synth.make_layer(spec, 3, seed, 4, 4, "bernoulli", 0.4)
        del lay
        lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, dtype)
        ref = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, dtype)(xs[0].clone())
        assert torch.equal(lay(xs[0], ys[0]), ref)


def test_layer_call_refuses_what_the_descriptor_refuses():
    spec = synth.ConvSpec("l", 16, 16, (1, 1, 1), (1, 1, 1), (0, 0, 0), True)
    L = synth.make_layer(spec, 3, 0, 4, 4, "none", None)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], None, dense=True)
    x = torch.zeros((1, 2, 4, 4, 16), dtype=torch.bfloat16, device="cuda")
    for bad, err in ((x[0], ValueError), (x.transpose(2, 3)[:, :, :2], ValueError), (x.half(), KeyError),
                     (x[..., :8].contiguous(), rt3d.Rt3dError)):
        with pytest.raises(err):
            lay(bad, torch.zeros_like(x))
    with pytest.raises(rt3d.Rt3dError):
        lay(x, x)                                                 # overlapping buffers


@pytest.mark.parametrize("name,clip", [("c3d", (16, 112, 112, 3)), ("r2plus1d", (4, 56, 56, 3)), ("s3d", (8, 96, 96, 3))])
def test_noted_forward_follows_a_bias_whose_storage_was_replaced(name, clip):
    net, _ = bench.build_network(name)
    x = nets.to_device(synth.make_input(9, (2,) + clip))
    before = net.forward(x).clone()
    old = []                                                      # the old storages stay in use
    for layer in net.layers.values():
        old.append(layer.bias.data)
        layer.bias.data = layer.bias.data + 0.25
    changed = net.forward(x).clone()
    assert not torch.equal(changed, before)
    assert torch.equal(changed, net._forward(x, 0, None, None))
    assert torch.equal(changed, net.forward(x))
    assert rt3d.rt3d_last_device_status() == rt3d.OK


@pytest.mark.parametrize("name,clip", [("c3d", (16, 112, 112, 3)), ("s3d", (8, 96, 96, 3))])
def test_noted_forward_writes_the_tensor_that_it_returns(name, clip):
    net, _ = bench.build_network(name)
    x = nets.to_device(synth.make_input(9, (2,) + clip))
    y = net.forward(x)
    want, old = y.clone(), y.data                                 # the old storage stays in use
    y.data = torch.zeros_like(y)
    again = net.forward(x)
    assert torch.equal(again, want)
    assert again.data_ptr() == y.data_ptr() != old.data_ptr()


@pytest.mark.parametrize("name,clip", [("c3d", (16, 112, 112, 3)), ("r2plus1d", (4, 56, 56, 3)), ("s3d", (8, 96, 96, 3))])
def test_noted_forward_refuses_a_freed_layer(name, clip):
    """A handle freed by hand is refused by the next pass, as a layer's own call refuses it; one that nobody uses, or that
    went with its last reference, leaves the notes alone."""
    net, _ = bench.build_network(name)
    x = nets.to_device(synth.make_input(9, (1,) + clip))
    want = net.forward(x).clone()
    noted = list(net._noted.values())
    spec = synth.ConvSpec("l", 16, 16, (1, 1, 1), (1, 1, 1), (0, 0, 0), True)
    L = synth.make_layer(spec, 3, 0, 4, 4, "none", None)
    for by_hand in (True, False):
        other = rt3d.rt3d_pack_dense(L["w"], rt3d.RT3D_BF16)
        if by_hand:
            other.free()
        del other
        assert torch.equal(net.forward(x), want)
        assert [a[0] for a in net._noted.values()] == [a[0] for a in noted]
    list(net.layers.values())[-1].packed.free()
    for _ in range(2):
        with pytest.raises(rt3d.Rt3dError) as e:
            net.forward(x)
        assert e.value.status == rt3d.ERR_INVALID_ARG
    torch.cuda.synchronize()


def test_small_copies_in_one_launch():
    """As many as a launch takes, one more, and lengths around a block's threads; values beside a destination stay."""
    src = torch.randn(70 * 300, device="cuda")
    dst = torch.full((70 * 301,), 7.0, device="cuda")
    for n in (1, 64, 65, 70):
        out, want, copies = dst.clone(), dst.clone(), []
        for i in range(n):
            count = (1, 255, 256, 257, 300)[i % 5]
            s = None if i % 7 == 3 else src[300 * i: 300 * i + count]
            copies.append((s, out, 301 * i, count))
            want[301 * i: 301 * i + count] = 0 if s is None else s
        launches = rt3d.rt3d_launch_count()
        rt3d.rt3d_copy_f32(copies)
        assert rt3d.rt3d_launch_count() - launches == -(-n // 64)
        assert torch.equal(out, want)
    for bad in ([], [(src, dst, 0, 0)]):
        with pytest.raises(rt3d.Rt3dError) as e:
            rt3d.rt3d_copy_f32(bad)
        assert e.value.status == rt3d.ERR_INVALID_ARG
