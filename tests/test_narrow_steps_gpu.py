"""Layers of up to 32 input channels in K steps of 32 (64-byte rows): the step-list kernels at their bundle widths, with one, two and
more steps, split along K, with temporal taps that share an input tile, strided, with a residual and through the dense entry, against
the oracle at the bf16 tolerance; and the same layers in steps of 64, which sum the same products in the same order."""
import numpy as np
import pytest
import torch

import oracle
import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu

PAIR, SINGLE = rt3d.ALGO_UMMA_PAIR, rt3d.ALGO_UMMA


@pytest.mark.parametrize("x,cin,cout,k,stride,kind,algo", [
    ((1, 2, 5, 7), 9, 16, (1, 1, 1), (1, 1, 1), "bernoulli", PAIR),                 # one step, the narrowest bundle
    ((2, 3, 9, 11), 16, 33, (3, 3, 3), (1, 1, 1), "bernoulli", SINGLE),
    ((1, 3, 9, 11), 17, 200, (3, 3, 3), (1, 1, 1), "bernoulli", SINGLE),            # a K split over a cluster
    ((1, 2, 7, 7), 31, 256, (3, 3, 3), (1, 1, 1), "bernoulli", SINGLE),             # ... with the widest share
    ((2, 4, 9, 11), 32, 130, (1, 3, 3), (1, 2, 2), "bernoulli", PAIR),              # two steps a stage, strided
    ((2, 4, 16, 16), 24, 64, (1, 3, 3), (1, 1, 1), "none", PAIR),                   # two issuing threads; the dense entry
    ((2, 8, 16, 16), 24, 96, (3, 3, 3), (1, 1, 1), "bernoulli", PAIR),              # taps share an input tile
    ((2, 8, 12, 12), 19, 240, (3, 3, 3), (1, 1, 1), "bernoulli", PAIR),
    ((1, 9, 12, 12), 20, 48, (7, 1, 1), (2, 1, 1), "bernoulli", PAIR),              # ... in two phases of a temporal stride
    ((3, 6, 13, 9), 30, 300, (3, 3, 3), (1, 1, 1), "exact_total", PAIR)])           # two bundles, one of them nearly empty
def test_steps_of_32_channels(x, cin, cout, k, stride, kind, algo):
    spec = synth.ConvSpec("n", cin, cout, k, stride, tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 13, cin + cout, 4, 4, kind, {"bernoulli": 0.5, "none": None, "exact_total": 7}[kind])
    xs = synth.make_input(13, x + (cin,))
    res = oracle.bf16_round(synth.make_input(14, (x[0],) + spec.out_extent(*x[1:]) + (cout,)))
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.bfloat16, dense=kind == "none")
    xd, rd = nets.to_device(xs, torch.bfloat16), nets.to_device(res, torch.bfloat16)
    conv = oracle.conv3d(xs, L["w"], L["mask"], L["bias"], spec.stride, spec.pad, False, round_bf16=True)
    for residual in (False, True):
        out = {}
        for narrow in (0, 1):
            rt3d.rt3d_debug_set(rt3d.DEBUG_NARROW, narrow)
            try:
                y = lay.fused(xd, lay.alloc_out(xd), residual=rd, algo=algo) if residual else lay(xd, algo=algo)
            finally:
                rt3d.rt3d_debug_set(rt3d.DEBUG_NARROW, 1)
            assert rt3d.rt3d_last_device_status() == rt3d.OK
            few = algo == SINGLE and k[0] * k[1] * k[2] <= 12          # few locations on single CTAs: steps of 64
            assert rt3d.rt3d_debug_get(rt3d.DEBUG_STEP_CHANNELS) == (32 if narrow and not few else 64)
            out[narrow] = nets.to_numpy(y, cout)
        ref = np.maximum(conv + (res if residual else 0), 0)
        assert np.abs(out[1] - ref).max() <= 2e-2 * np.abs(ref).max()
        assert np.abs(out[1] - out[0]).max() <= 2 ** -7 * np.abs(ref).max()      # a rounding apart at most: other K splits
