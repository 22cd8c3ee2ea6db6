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


CALLS = [  # channels in and out, kernel, stride, extents, type, family, residual: every kernel that a call can be prepared for
    (64, 64, (3, 3, 3), (1, 1, 1), (1, 4, 20, 20), torch.bfloat16, rt3d.ALGO_AUTO, True),
    (64, 64, (3, 3, 3), (1, 1, 1), (1, 4, 20, 20), torch.bfloat16, rt3d.ALGO_UMMA, False),
    (64, 96, (3, 3, 3), (1, 1, 1), (2, 4, 20, 20), torch.bfloat16, rt3d.ALGO_UMMA_PAIR, True),
    (32, 64, (1, 3, 3), (1, 1, 1), (1, 4, 16, 16), torch.bfloat16, rt3d.ALGO_UMMA_HALO, True),
    (64, 64, (3, 3, 3), (1, 1, 1), (1, 4, 12, 12), torch.bfloat16, rt3d.ALGO_UMMA_SUB, True),
    (64, 40, (3, 3, 3), (1, 1, 1), (1, 4, 12, 12), torch.bfloat16, rt3d.ALGO_SIMT, True),
    (3, 45, (1, 7, 7), (1, 2, 2), (1, 4, 32, 32), torch.bfloat16, rt3d.ALGO_AUTO, True),
    (3, 64, (3, 3, 3), (1, 1, 1), (1, 4, 24, 24), torch.bfloat16, rt3d.ALGO_AUTO, True),
    (24, 40, (3, 3, 3), (1, 1, 1), (1, 4, 12, 12), torch.float32, rt3d.ALGO_AUTO, True)]


@pytest.mark.parametrize("cin,cout,k,stride,ext,dtype,algo,res", CALLS)
def test_prepared_call_on_buffers_it_has_not_seen(cin, cout, k, stride, ext, dtype, algo, res):
    """A call is prepared for its shapes, not for its buffers: new ones give the bits of a handle that has prepared nothing,
    with and without a bias, and what depends on an address is refused as on a first call."""
    spec = synth.ConvSpec("l", cin, cout, k, stride, tuple(a // 2 for a in k), True)
    L = synth.make_layer(spec, 3, 0, 4, 4, "bernoulli", 0.5)
    make = lambda: nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, dtype)

    def call(lay, x, y, r):
        return lay.fused(x, y, residual=r, algo=algo) if r is not None else lay(x, y, algo=algo)

    def shifted(t, n=1):                                          # the same values 16 n bytes further on
        flat = torch.zeros(t.numel() + 256, dtype=t.dtype, device="cuda")
        at = n * 16 // t.element_size()
        flat[at: at + t.numel()] = t.flatten()
        return flat[at: at + t.numel()].view(t.shape)

    lay = make()
    for i in range(6):
        x = shifted(nets.to_device(synth.make_input(i, ext + (cin,)), dtype), i)
        y = shifted(torch.zeros(lay.out_shape(x), dtype=dtype, device="cuda"), 2 * i)
        r = None
        if res and i != 3:
            r = shifted(torch.zeros_like(y), i + 1)
            r[..., :cout] = torch.randn(r[..., :cout].shape, device="cuda")
        want = torch.zeros_like(y)
        other = make()
        if i == 4:
            lay.bias = other.bias = None
        elif i == 5:
            lay.bias = other.bias = torch.randn(cout, device="cuda")
        call(other, x, want, r)
        call(lay, x, y, r)
        assert torch.equal(y, want), i
    flat = torch.zeros(x.numel() + 64, dtype=dtype, device="cuda")
    bad_x = flat[1: 1 + x.numel()].view(x.shape)                  # off the 16-byte boundary
    flat = torch.zeros(y.numel() + 64, dtype=dtype, device="cuda")
    bad_y = flat[1: 1 + y.numel()].view(y.shape)
    both = torch.zeros(max(x.numel(), y.numel()), dtype=dtype, device="cuda")
    over_x, over_y = both[: x.numel()].view(x.shape), both[: y.numel()].view(y.shape)
    bad = [(bad_x, y, r), (x, bad_y, r), (over_x, over_y, r)]
    if res:
        bad += [(x, y, y), (x, y, bad_y)]
    for args in bad:
        launches = rt3d.rt3d_launch_count()
        with pytest.raises(rt3d.Rt3dError) as e:
            call(lay, *args)
        assert e.value.status == rt3d.ERR_INVALID_ARG and rt3d.rt3d_launch_count() == launches
    assert rt3d.rt3d_last_device_status() == rt3d.OK


def test_prepared_pair_on_buffers_it_has_not_seen():
    s = synth.ConvSpec("s", 64, 144, (1, 3, 3), (1, 1, 1), (0, 1, 1), True)
    t = synth.ConvSpec("t", 144, 64, (3, 1, 1), (1, 1, 1), (1, 0, 0), True)
    ls, lt = (synth.make_layer(sp, 3, i, 4, 4, "bernoulli", 0.4) for i, sp in enumerate((s, t)))
    make = lambda: [nets.ConvLayer(sp, L["w"], L["bias"], L["mask"]) for sp, L in ((s, ls), (t, lt))]

    def call(pair, x, y, r, biases=(True, True)):
        rt3d.rt3d_conv2plus1d_fused(rt3d.tensor_desc(x), pair[0].packed, pair[0].bias if biases[0] else None, s.pad, True,
                                    pair[1].packed, pair[1].bias if biases[1] else None, t.pad, True, rt3d.tensor_desc(y),
                                    None if r is None else rt3d.tensor_desc(r))

    pair = make()
    for i in range(6):
        x = nets.to_device(synth.make_input(i, (1, 4, 24, 24, 64)))
        y, want = torch.zeros_like(x), torch.zeros_like(x)
        r = torch.randn_like(x) if i % 2 else None
        biases = (i != 4, i != 5)
        call(make(), x, want, r, biases)
        call(pair, x, y, r, biases)
        assert torch.equal(y, want), i
    assert rt3d.rt3d_last_plan()["kernel"] == 5
    with pytest.raises(rt3d.Rt3dError):
        call(pair, x, x, None)
    assert rt3d.rt3d_last_device_status() == rt3d.OK
