"""Epilogue pieces that are turned in shared memory (layers with a residual, and tiles that box stores cannot take): channel counts
around the 16-byte units and the 32-channel pieces, boxes of every kind, a residual whose padding holds NaNs, and padding
channels of the output that must stay as they are.  Against the oracle at the bf16 tolerance of the other tests."""
import numpy as np
import pytest
import torch

import oracle
import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import binding, nets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x,cin,cout,k,stride,algo,residual", [
    ((2, 4, 9, 11), 40, 64, (3, 3, 3), (1, 1, 1), rt3d.ALGO_UMMA_PAIR, True),       # boxes that are not whole blocks of 32
    ((2, 4, 9, 11), 40, 65, (3, 3, 3), (1, 1, 1), rt3d.ALGO_UMMA_PAIR, True),       # 80 columns: a piece of 16, one channel in a unit
    ((2, 4, 9, 11), 40, 95, (3, 3, 3), (1, 1, 1), rt3d.ALGO_UMMA_PAIR, False),      # seven channels in the last unit
    ((1, 5, 13, 7), 70, 150, (1, 3, 3), (1, 2, 2), rt3d.ALGO_UMMA_PAIR, False),
    ((2, 4, 16, 16), 64, 128, (3, 3, 3), (1, 1, 1), rt3d.ALGO_UMMA_PAIR, True),     # box stores, two issuing threads
    ((2, 4, 16, 16), 64, 250, (1, 3, 3), (1, 1, 1), rt3d.ALGO_UMMA_PAIR, True),     # the last piece ends in two channels
    ((3, 3, 7, 5), 64, 300, (3, 1, 1), (1, 1, 1), rt3d.ALGO_UMMA_PAIR, True),       # two bundles, an odd number of tiles
    ((2, 3, 17, 9), 64, 100, (1, 3, 3), (1, 1, 1), rt3d.ALGO_UMMA_HALO, True),      # 16 x 8 tiles that hang over
    ((2, 3, 16, 8), 33, 64, (1, 1, 1), (1, 1, 1), rt3d.ALGO_UMMA_HALO, True)])
def test_turned_pieces(x, cin, cout, k, stride, algo, residual):
    spec = synth.ConvSpec("t", cin, cout, k, stride, tuple(v // 2 for v in k), True)
    L = synth.make_layer(spec, 12, cin + cout, 4, 4, "bernoulli", 0.5)
    xs = synth.make_input(12, x + (cin,))
    conv = oracle.conv3d(xs, L["w"], L["mask"], L["bias"], spec.stride, spec.pad, False, round_bf16=True)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.bfloat16)
    xd = nets.to_device(xs, torch.bfloat16)
    y = torch.full(lay.out_shape(xd)[:4] + (nets.pitch_for(cout, torch.bfloat16) + 16,), 55.0, dtype=torch.bfloat16, device="cuda")
    res = None
    if residual:
        res = torch.full_like(y, float("nan"))
        res[..., :cout] = torch.rand(y.shape[:4] + (cout,), device="cuda") * 2 - 1
        conv = conv.astype(np.float64) + res[..., :cout].float().cpu().numpy()
    ref = np.maximum(conv, 0)
    with binding.concurrent_kernels():                     # whole tiles only, no tail split
        rt3d.rt3d_conv3d_sparse_fused(rt3d.tensor_desc(xd, cin), lay.packed, lay.bias, rt3d.tensor_desc(y, cout), spec.stride, spec.pad,
                                      True, residual=rt3d.tensor_desc(res, cout) if residual else None, algo=algo)
    assert rt3d.rt3d_last_device_status() == rt3d.OK
    assert rt3d.rt3d_last_plan()["kernel"] == 4 if algo == rt3d.ALGO_UMMA_HALO else rt3d.rt3d_last_plan()["kernel"] in (2, 7)
    assert rt3d.rt3d_last_plan()["tail_workers"] == 0 and rt3d.rt3d_debug_get(rt3d.DEBUG_TURNED) == 1
    got = y.float().cpu().numpy()
    assert np.abs(got[..., :cout] - ref).max() <= 2e-2 * np.abs(ref).max()
    unit = (cout + 7) // 8 * 8                             # box stores may zero the rest of a row's last 16-byte unit
    assert (got[..., unit:] == 55.0).all()


@pytest.mark.parametrize("cin,cout,k", [(64, 128, (3, 3, 3)), (83, 150, (3, 3, 3))])
def test_turned_tiles_beside_a_tail_split(cin, cout, k):
    """Whole rounds of tiles, which are turned, and a last one that is shared out along K, which is not."""
    spec = synth.ConvSpec("t", cin, cout, k, (1, 1, 1), (1, 1, 1), True)
    L = synth.make_layer(spec, 12, cin + cout, 4, 4, "bernoulli", 0.5)
    lay = nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.bfloat16)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for clips in range(8, 64):                             # 100 tiles a clip: look for a count with a shared last round
        x = (clips, 8, 40, 40)
        xd = torch.zeros(x + (nets.pitch_for(cin, torch.bfloat16),), dtype=torch.bfloat16, device="cuda")
        y = lay.alloc_out(xd)
        with rt3d.planning():
            lay.fused(xd, y, residual=y.new_zeros(y.shape))
        plan = rt3d.rt3d_last_plan()
        if plan["tail_workers"] > 0 and rt3d.rt3d_debug_get(rt3d.DEBUG_TURNED) == 1:
            break
    assert plan["tail_workers"] > 0 and plan["kernel"] in (2, 7) and clips * 100 > sms
    gen = torch.Generator(device="cuda").manual_seed(2)
    xd[..., :cin] = (torch.rand(x + (cin,), device="cuda", generator=gen) * 2 - 1).bfloat16()
    res = torch.full_like(y, float("nan"))
    res[..., :cout] = (torch.rand(y.shape[:4] + (cout,), device="cuda", generator=gen) * 2 - 1).bfloat16()
    rt3d.rt3d_conv3d_sparse_fused(rt3d.tensor_desc(xd, cin), lay.packed, lay.bias, rt3d.tensor_desc(y, cout), spec.stride, spec.pad, True,
                                  residual=rt3d.tensor_desc(res, cout))
    assert rt3d.rt3d_last_plan() == plan and rt3d.rt3d_last_device_status() == rt3d.OK and rt3d.rt3d_debug_get(rt3d.DEBUG_TURNED) == 1
    want = torch.relu(lay(xd, relu=False, algo=rt3d.ALGO_SIMT)[..., :cout].float() + res[..., :cout].float())
    got = y[..., :cout].float()
    assert float((got - want).abs().max()) <= 2e-2 * float(want.abs().max())
