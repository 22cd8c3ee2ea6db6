"""Register-blocked fp32 convolution kernel: shapes at the edges of its boxes, row sets, stages and quads, against the
oracle.  fp32 FMAs in another order than the oracle's double sums: 2e-6 of the largest output is about twice what the
longest sum here shows."""
import numpy as np
import pytest
import torch

import oracle
import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x,cin,cout,k,stride,group,kind,density", [
    ((1, 8, 28, 28), 16, 32, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.5),       # whole sets and quads
    ((1, 1, 1, 1), 4, 4, (1, 1, 1), (1, 1, 1), (4, 4), "none", None),               # the smallest call
    ((2, 3, 5, 7), 1, 1, (3, 3, 3), (1, 1, 1), (4, 4), "none", None),               # one channel each way
    ((3, 5, 9, 11), 37, 43, (3, 3, 3), (2, 2, 2), (4, 4), "bernoulli", 0.4),        # ragged channels and extents, strided
    ((1, 4, 33, 31), 30, 130, (1, 3, 3), (1, 2, 2), (8, 4), "bernoulli", 0.3),      # a row set beyond 128 outputs
    ((2, 9, 17, 5), 70, 33, (3, 1, 1), (1, 1, 1), (8, 8), "bernoulli", 0.2),        # four quads a stage, groups of two quads
    ((2, 6, 14, 13), 34, 65, (1, 1, 1), (2, 2, 2), (4, 4), "bernoulli", 0.4),       # eight quads a stage, sampled input
    ((1, 4, 20, 20), 12, 40, (1, 7, 7), (1, 2, 2), (4, 4), "bernoulli", 0.4),       # 49 locations
    ((1, 2, 6, 6), 64, 512, (3, 3, 3), (1, 1, 1), (8, 4), "vanilla_total", 200),    # whole groups: empty and full stages
    ((1, 2, 6, 6), 24, 40, (3, 3, 3), (1, 1, 1), (4, 4), "exact_total", 1),         # one place kept in all
    ((1, 4, 14, 14), 61, 122, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.4),      # few voxels: warps that share them
    ((1, 2, 7, 7), 128, 128, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.05),      # ... with parts of nearly empty lists
    ((4, 16, 40, 40), 16, 128, (3, 3, 3), (1, 1, 1), (4, 4), "bernoulli", 0.4)])    # several boxes per SM
def test_fp32_kernel_matches_oracle(x, cin, cout, k, stride, group, kind, density):
    spec = synth.ConvSpec("f32", cin, cout, k, stride, tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 8, cin + cout, group[0], group[1], kind, density)
    xs = synth.make_input(8, x + (cin,))
    to = spec.out_extent(*x[1:])
    res = synth.uniform_pm1(77, (x[0],) + to + (cout,))
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], group[0], group[1], torch.float32, dense=kind == "none")
    xd = nets.to_device(xs, torch.float32)
    xd[..., cin:] = float("nan")                           # padding channels of the input are never read as data
    y = torch.full(lay.out_shape(xd), 3.0, device="cuda")
    for residual in (None, res):
        if residual is None:
            lay(xd, y, relu=False)
        else:
            lay.fused(xd, y, residual=nets.to_device(res, torch.float32), relu=True)
        assert rt3d.rt3d_last_plan()["kernel"] == 0 and rt3d.rt3d_last_device_status() == rt3d.OK
        ref = oracle.conv3d(xs, L["w"], L["mask"], L["bias"], spec.stride, spec.pad, False)
        if residual is not None:
            ref = np.maximum(ref + res, 0.0)
        got = y.cpu().numpy()
        assert np.abs(got[..., :cout] - ref).max() <= 2e-6 * np.abs(ref).max()
        assert (got[..., cout:] == 3.0).all()              # those of the output are not written
