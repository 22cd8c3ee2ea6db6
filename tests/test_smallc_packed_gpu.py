"""Small-C_in kernel with two input columns per entry (at most four channels, column stride 2): even and odd kernel widths,
pruned locations, extents that cut the 16 x 8 tile, row and frame strides, the caller's padding channels NaN."""
import numpy as np
import pytest
import torch

import oracle
import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x,cin,cout,k,stride,density", [
    ((1, 3, 33, 17), 3, 45, (1, 7, 7), (1, 2, 2), 0.5),
    ((2, 2, 31, 35), 3, 64, (1, 7, 7), (1, 2, 2), 1.0),
    ((1, 5, 20, 18), 4, 64, (3, 4, 4), (2, 2, 2), 0.5),
    ((1, 4, 9, 40), 1, 16, (3, 3, 3), (1, 1, 2), 0.5),
    ((1, 2, 16, 16), 2, 24, (1, 5, 2), (1, 3, 2), 0.7),
    ((1, 3, 34, 34), 3, 128, (2, 3, 5), (1, 2, 2), 0.1)])
def test_packed_small_cin_matches_oracle(x, cin, cout, k, stride, density):
    spec = synth.ConvSpec("sc", cin, cout, k, stride, tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 77, cin + cout, 4, 4, "bernoulli", density)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.bfloat16)
    xs = synth.make_input(770, x + (cin,))
    xd = nets.to_device(xs)
    xd[..., cin:] = float("nan")
    y = torch.zeros(lay.out_shape(xd), dtype=torch.bfloat16, device="cuda")
    lay.fused(xd, y)
    assert rt3d.rt3d_last_plan()["kernel"] == 3
    ref = np.maximum(oracle.conv3d(xs, L["w"], L["mask"], L["bias"], spec.stride, spec.pad, False, round_bf16=True), 0.0)
    assert rt3d.rt3d_last_device_status() == rt3d.OK
    assert np.abs(nets.to_numpy(y, cout) - ref).max() <= 2e-2 * np.abs(ref).max()
