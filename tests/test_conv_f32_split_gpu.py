"""fp32 convolution on the tensor cores (plan kernel 8: every value as three bf16 ones) against the oracle, at the edges of its
tiles, chunks, bundle widths and accumulator periods.

Tolerance: a product of two values split three ways is wrong by less than 2^-23 of it, the sums are fp32 over at most 8 steps of
32 channels and fp32 from there on: 2e-6 of the largest output, as for the CUDA-core kernel, is several times what the longest
sum here shows."""
import numpy as np
import pytest
import torch

import oracle
import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


@pytest.fixture
def everywhere():
    rt3d.rt3d_debug_set(rt3d.DEBUG_F32_SPLIT, 2)
    yield
    rt3d.rt3d_debug_set(rt3d.DEBUG_F32_SPLIT, 1)


@pytest.mark.parametrize("x,cin,cout,k,stride,group,kind,density", [
    ((1, 1, 1, 1), 4, 4, (1, 1, 1), (1, 1, 1), (4, 4), "none", None),               # one voxel, one step of half a chunk
    ((1, 8, 28, 28), 16, 32, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.5),       # 16 channels: half chunks only; 32 columns
    ((2, 3, 9, 11), 17, 33, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.4),        # just above both; ragged outputs, 48 columns
    ((3, 5, 9, 11), 37, 43, (3, 3, 3), (2, 2, 2), (4, 4), "bernoulli", 0.4),        # a last chunk of half; strided; odd step count
    ((2, 4, 16, 16), 64, 64, (1, 3, 3), (1, 2, 2), (8, 4), "bernoulli", 0.3),       # 64 columns: shared small products
    ((1, 4, 33, 31), 30, 65, (1, 3, 3), (1, 1, 1), (8, 4), "bernoulli", 0.3),       # pairs: 80 columns, the second set of 32
    ((2, 9, 17, 5), 70, 96, (3, 1, 1), (1, 1, 1), (8, 8), "bernoulli", 0.2),        # 96 columns, an odd number of tiles
    ((2, 6, 14, 13), 34, 97, (1, 1, 1), (2, 2, 2), (4, 4), "none", None),           # 112 columns, one step a hand-shake
    ((1, 6, 20, 20), 96, 128, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.4),      # 81 steps: more than one segment of 64
    ((1, 5, 12, 12), 70, 150, (3, 3, 3), (1, 1, 1), (3, 5), "bernoulli", 0.4),      # two bundles; groups that no other fp32 kernel blocks
    ((1, 2, 6, 6), 64, 256, (3, 3, 3), (1, 1, 1), (8, 4), "vanilla_total", 40),     # bundles with few steps
    ((1, 2, 6, 6), 24, 40, (3, 3, 3), (1, 1, 1), (4, 4), "exact_total", 1),         # one place kept in all
    ((2, 2, 6, 6), 64, 200, (3, 3, 3), (1, 1, 1), (8, 8), "exact_total", 1),        # a bundle without any step
    ((5, 16, 40, 40), 33, 48, (3, 1, 1), (1, 1, 1), (4, 4), "bernoulli", 0.4)])     # several items per SM
def test_split_kernel_matches_oracle(everywhere, x, cin, cout, k, stride, group, kind, density):
    spec = synth.ConvSpec("f32", cin, cout, k, stride, tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 8, cin + cout, group[0], group[1], kind, density)
    xs = synth.make_input(8, x + (cin,))
    res = synth.uniform_pm1(77, (x[0],) + spec.out_extent(*x[1:]) + (cout,))
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], group[0], group[1], torch.float32, dense=kind == "none")
    xd = nets.to_device(xs, torch.float32)
    xd[..., cin:] = float("nan")                           # padding channels of the input are never read as data
    y = torch.full(lay.out_shape(xd), 3.0, device="cuda")
    for residual in (None, res):
        if residual is None:
            lay(xd, y, relu=False)
        else:
            lay.fused(xd, y, residual=nets.to_device(res, torch.float32), relu=True)
        assert rt3d.rt3d_last_plan()["kernel"] == 8 and rt3d.rt3d_last_device_status() == rt3d.OK
        ref = oracle.conv3d(xs, L["w"], L["mask"], L["bias"], spec.stride, spec.pad, False)
        if residual is not None:
            ref = np.maximum(ref + res, 0.0)
        got = y.cpu().numpy()
        assert np.abs(got[..., :cout] - ref).max() <= 2e-6 * np.abs(ref).max()
        assert (got[..., cout:] == 3.0).all()              # those of the output are not written


@pytest.mark.parametrize("cin,cout", [(40, 24), (40, 64), (40, 120)])
def test_values_that_three_bf16_cannot_hold(everywhere, cin, cout):
    """Infinities, NaNs, values next to the largest float and tiny ones: every output is what the CUDA-core kernel gives, up to
    the order of its sums, and what pruned weights would have met has no effect."""
    spec = synth.ConvSpec("f32", cin, cout, (3, 3, 3), (1, 1, 1), (1, 1, 1), False)
    L = synth.make_layer(spec, 9, cin + cout, 4, 4, "bernoulli", 0.3)
    xs = synth.make_input(9, (2, 4, 12, 12, cin))
    xs[0, 1, 3, 4, 5] = np.inf
    xs[0, 2, 8, 8, 21] = -np.inf
    xs[0, 3, 10, 1, 7] = np.nan
    xs[1, 0, 2, 2, 11] = 3.4e38
    xs[1, 2, 6:, 6:, :] *= np.float32(1e-33)               # windows of nothing else: tiny outputs
    xs[1, 1, 6:, 6:, :] *= np.float32(1e-33)
    xs[1, 3, 6:, 6:, :] *= np.float32(1e-33)
    lay = nets.ConvLayer(spec, L["w"], np.zeros_like(L["bias"]), L["mask"], 4, 4, torch.float32)
    xd = nets.to_device(xs, torch.float32)
    got = lay(xd).cpu().numpy()
    assert rt3d.rt3d_last_plan()["kernel"] == 8 and rt3d.rt3d_last_device_status() == rt3d.OK
    want = lay(xd, algo=rt3d.ALGO_SIMT).cpu().numpy()
    assert rt3d.rt3d_last_plan()["kernel"] == 0
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.isnan(want).any()
    assert np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
    assert np.isinf(want).any()
    rows = np.isfinite(want).all(axis=-1)                  # a voxel's sums are as wrong as its largest ones
    err, size = np.abs(got[rows] - want[rows]).max(axis=-1), np.abs(want[rows]).max(axis=-1)
    assert (size[size > 0].min() < 1e-32) and (err <= 1e-5 * size).all()


def test_weights_that_three_bf16_cannot_hold_stay_on_the_cuda_cores(everywhere):
    spec = synth.ConvSpec("f32", 32, 32, (1, 3, 3), (1, 1, 1), (0, 1, 1), False)
    L = synth.make_layer(spec, 9, 1, 4, 4, "none", None)
    xd = nets.to_device(synth.make_input(9, (1, 2, 8, 8, 32)), torch.float32)
    for value in (1e-31, 3e36, np.inf, np.nan, -0.0):
        w = L["w"].copy()
        w[3, 5, 0, 1, 1] = value
        nets.ConvLayer(spec, w, L["bias"], None, 4, 4, torch.float32, dense=True)(xd)
        assert rt3d.rt3d_last_plan()["kernel"] == (8 if value == 0.0 else 0)


@pytest.mark.parametrize("cin,cout,k,x", [
    (64, 64, (3, 3, 3), (2, 8, 40, 40)), (64, 16, (3, 3, 3), (2, 8, 40, 40)), (96, 90, (3, 3, 3), (2, 8, 40, 40)),
    (20, 3000, (1, 1, 1), (1, 2, 6, 6)), (20, 7680, (1, 1, 1), (1, 2, 6, 6))])           # biases that leave three weight stages, two inputs
def test_inputs_that_arrive_late(everywhere, cin, cout, k, x):
    """Boxes from memory beside boxes in the padding, which take no load at all: with nothing in L2 every pass gives the same bits,
    and what the CUDA cores give up to the order of the sums."""
    spec = synth.ConvSpec("f32", cin, cout, k, (1, 1, 1), tuple(v // 2 for v in k), False)
    L = synth.make_layer(spec, 8, cin + cout, 4, 4, "bernoulli", 0.4)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.float32)
    xd = nets.to_device(synth.make_input(8, x + (cin,)), torch.float32)
    want = lay(xd, algo=rt3d.ALGO_SIMT)
    flush = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    first = lay(xd)
    assert rt3d.rt3d_last_plan()["kernel"] == 8
    assert float((first - want).abs().max()) <= 2e-6 * float(want.abs().max())
    for i in range(5):
        flush.fill_(i)
        assert torch.equal(lay(xd), first) and rt3d.rt3d_last_device_status() == rt3d.OK


@pytest.mark.parametrize("cin,cout", [(40, 24), (40, 120)])
@pytest.mark.parametrize("x_exp,w_exp", [(-115, 0), (-120, 0), (-130, 0), (-140, 0), (-147, 0), (-120, 40), (-128, 60), (-140, 60),
                                         (-149, 63), (-60, -75), (60, 0), (90, 4), (120, 0), (-130, 100), (-136, 119)])
def test_magnitudes_at_both_ends_of_the_range(everywhere, cin, cout, x_exp, w_exp):
    """Inputs down to the smallest denormal and weights up to the largest: against sums in 64 bits, with the error of ordinary
    magnitudes and that of a few roundings of a denormal result.  Handles whose weights do not fit run on the CUDA cores."""
    spec = synth.ConvSpec("f32", cin, cout, (1, 3, 3), (1, 1, 1), (0, 1, 1), False)
    L = synth.make_layer(spec, 9, cin + cout, 4, 4, "bernoulli", 0.4)
    w = np.ldexp(L["w"] / np.float32(np.abs(L["w"]).max()), w_exp).astype(np.float32)
    x = np.ldexp(synth.make_input(9, (1, 2, 8, 8, cin)), x_exp + 1).astype(np.float32)
    lay = nets.ConvLayer(spec, w, np.zeros_like(L["bias"]), L["mask"], 4, 4, torch.float32)
    got = lay(nets.to_device(x, torch.float32)).cpu().numpy()[..., :cout].astype(np.float64)
    assert rt3d.rt3d_last_plan()["kernel"] == (8 if w_exp < 64 else 0) and rt3d.rt3d_last_device_status() == rt3d.OK
    xp = np.pad(x.astype(np.float64), ((0, 0), (0, 0), (1, 1), (1, 1), (0, 0)))
    wm = (w * L["mask"]).astype(np.float64)
    ref = sum(xp[:, :, a:a + 8, b:b + 8] @ wm[:, :, 0, a, b].T for a in range(3) for b in range(3))
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max() + 40 * 9 * 2.0 ** -150


@pytest.mark.parametrize("cin,cout,group,share", [
    (64, 128, (4, 4), 1.0), (40, 90, (8, 8), 1.0), (37, 51, (3, 5), 1.0), (33, 64, (1, 1), 0.5), (70, 24, (8, 3), 0.5), (30, 100, (8, 6), 1.0),
    (606, 128, (1, 1), 1.0)])                              # the last: as much as a warp may have to do again for a tile
def test_tiles_of_rows_that_are_computed_again(everywhere, cin, cout, group, share):
    """An input of infinities and NaNs: every row is computed again, by whichever lanes, as the CUDA cores do it, with a residual
    and ragged channels, and the roles that wait for it do not give up."""
    spec = synth.ConvSpec("f32", cin, cout, (3, 3, 3) if cin > 600 else (1, 3, 3), (1, 1, 1), (1, 1, 1) if cin > 600 else (0, 1, 1), False)
    L = synth.make_layer(spec, 9, cin + cout, group[0], group[1], "bernoulli", 0.9 if cin > 600 else 0.3)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], group[0], group[1], torch.float32)
    xd = nets.to_device(synth.make_input(9, (2, 2, 10, 10, cin)), torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(1)
    hit = torch.rand(xd.shape, device="cuda", generator=gen) < 0.002 * share
    xd[hit] = float("inf")
    xd[:, :, 5:] = torch.where(torch.rand(xd[:, :, 5:].shape, device="cuda", generator=gen) < share, xd[:, :, 5:] * 1e37, xd[:, :, 5:])
    xd[0, 1, 2, 3, 4] = float("nan")
    xd[..., cin:] = float("nan")
    res = torch.rand(lay.out_shape(xd), device="cuda", generator=gen)
    got, want = torch.full(lay.out_shape(xd), 3.0, device="cuda"), torch.full(lay.out_shape(xd), 3.0, device="cuda")
    lay.fused(xd, got, residual=res, relu=False)
    assert rt3d.rt3d_last_plan()["kernel"] == 8 and rt3d.rt3d_last_device_status() == rt3d.OK
    rt3d.rt3d_debug_set(rt3d.DEBUG_F32_SPLIT, 0)
    lay.fused(xd, want, residual=res, relu=False)
    assert rt3d.rt3d_last_plan()["kernel"] == 0
    assert (got[..., cout:] == 3.0).all()
    got, want = got[..., :cout].double(), want[..., :cout].double()
    assert torch.equal(got.isnan(), want.isnan()) and torch.equal(got.isposinf(), want.isposinf()) and torch.equal(got.isneginf(), want.isneginf())
    rows = want.isfinite().all(dim=-1)
    assert (rows.any() or cin > 600) and (~want.isfinite()).any()
    if rows.any():
        err, size = (got[rows] - want[rows]).abs().amax(dim=-1), want[rows].abs().amax(dim=-1)
        assert (err <= 1e-5 * size).all()


def test_layers_with_more_to_compute_again_stay_on_the_cuda_cores(everywhere):
    spec = synth.ConvSpec("f32", 608, 16, (3, 3, 3), (1, 1, 1), (1, 1, 1), False)
    x = torch.zeros((1, 1, 4, 4, 608), device="cuda")
    for group, kernel in (((1, 1), 0), ((2, 1), 8), ((4, 4), 8)):
        L = synth.make_layer(spec, 9, 1, group[0], group[1], "bernoulli", 0.05)
        nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], group[0], group[1], torch.float32)(x)
        assert rt3d.rt3d_last_plan()["kernel"] == kernel


@pytest.mark.parametrize("cin,cout,density,kernel", [(15, 118, None, 8), (16, 118, 0.9, 0), (17, 118, 0.9, 8)])
def test_layers_of_up_to_16_channels(cin, cout, density, kernel):
    """Half of a step is empty: the dispatch sends unpruned ones, and the results are the CUDA cores' up to the order of the sums."""
    spec = synth.ConvSpec("f32", cin, cout, (3, 3, 3), (1, 1, 1), (1, 1, 1), True)
    L = synth.make_layer(spec, 8, cin, 4, 4, "bernoulli" if density else "none", density)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.float32, dense=density is None)
    x = nets.to_device(synth.make_input(8, (3, 12, 28, 31, cin)), torch.float32)
    got = lay(x)
    assert rt3d.rt3d_last_plan()["kernel"] == kernel and rt3d.rt3d_last_device_status() == rt3d.OK
    want = lay(x, algo=rt3d.ALGO_SIMT)
    assert float((got - want).abs().max()) <= 2e-6 * float(want.abs().max())
