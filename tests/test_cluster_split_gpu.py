"""K split over a thread-block cluster (single-CTA kernel): every split count, bundle widths whose columns do not divide
evenly among the CTAs, ragged channels and voxels, residual, shares without steps; against the oracle, and repeatable."""
import numpy as np
import pytest
import torch

import oracle
import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x,cin,cout,k,density", [
    ((1, 2, 7, 7), 512, 512, (3, 3, 3), 0.3),          # one tile of 98 voxels
    ((1, 2, 7, 7), 512, 33, (3, 3, 3), 0.3),           # 48 columns: fewer units than CTAs
    ((1, 3, 9, 5), 256, 230, (3, 3, 3), 0.4),          # 240 columns, 135 voxels in two tiles
    ((2, 4, 14, 14), 256, 200, (1, 3, 3), 0.4),        # a split count that is no power of two
    ((8, 2, 7, 7), 1152, 512, (3, 1, 1), 0.4),
    ((8, 2, 7, 7), 512, 1152, (1, 3, 3), 0.4),
    ((1, 2, 5, 5), 640, 24, (1, 1, 3), 0.5),           # 32 columns and fewer
    ((16, 2, 7, 7), 512, 512, (3, 3, 3), None)])       # the dense path
def test_cluster_split_matches_oracle(x, cin, cout, k, density):
    spec = synth.ConvSpec("cl", cin, cout, k, (1, 1, 1), tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 61, cin + cout, 4, 4, "none" if density is None else "bernoulli", density)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.bfloat16, dense=density is None)
    xs = synth.make_input(610, x + (cin,))
    xd = nets.to_device(xs)
    ref0 = oracle.conv3d(xs, L["w"], L["mask"], L["bias"], spec.stride, spec.pad, False, round_bf16=True)
    res = synth.uniform_pm1(61, ref0.shape)
    rd = nets.to_device(res)
    for residual in (False, True):
        y = [torch.full(lay.out_shape(xd), 9.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        for v in y:
            lay.fused(xd, v, residual=rd if residual else None)
        plan = rt3d.rt3d_last_plan()
        assert plan["kernel"] == 1 and plan["n_splits"] > 1, plan
        assert rt3d.rt3d_last_device_status() == rt3d.OK and torch.equal(y[0], y[1])
        ref = np.maximum(ref0 + (oracle.bf16_round(res) if residual else 0.0), 0.0)
        assert np.abs(nets.to_numpy(y[0], cout) - ref).max() <= 2e-2 * np.abs(ref).max()
        assert (y[0][..., cout:] == 9.0).all()
