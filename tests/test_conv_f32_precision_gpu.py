"""fp32 layers against sums in 64 bits: the tensor-core kernel (every value as three bf16 ones) is no further off than the CUDA-core
kernel, for short and long sums, inputs of both signs and of one, and layers whose sums have one sign are not sent there."""
import itertools

import numpy as np
import pytest
import torch

import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


def _errors(cin, cout, k, density, x_one_sign, w_mean):
    """2-norm of the error over that of the result: the CUDA-core kernel's, the chosen kernel's, and which that is."""
    spec = synth.ConvSpec("f32", cin, cout, k, (1, 1, 1), tuple(v // 2 for v in k), False)
    L = synth.make_layer(spec, 8, cin + cout, 4, 4, "none" if density == 1.0 else "bernoulli", None if density == 1.0 else density)
    w = (np.abs(L["w"]) if w_mean == "one sign" else L["w"] + np.float32(w_mean * 0.05)).astype(np.float32)
    lay = nets.ConvLayer(spec, w, np.zeros_like(L["bias"]), L["mask"], 4, 4, torch.float32, dense=density == 1.0)
    gen = torch.Generator(device="cuda").manual_seed(cin)
    x = torch.zeros((2, 8, 28, 28, nets.pitch_for(cin, torch.float32)), device="cuda")
    x[..., :cin] = torch.rand(x.shape[:4] + (cin,), device="cuda", generator=gen)
    if not x_one_sign:
        x[..., :cin] = 2 * x[..., :cin] - 1
    wd = torch.from_numpy(w if L["mask"] is None else w * L["mask"]).cuda().double()
    xp = torch.nn.functional.pad(x[..., :cin].double(), [v // 2 for v in (1, 1, k[2], k[2], k[1], k[1], k[0], k[0])])
    ref = sum(xp[:, a:a + 8, b:b + 28, c:c + 28] @ wd[:, :, a, b, c].T for a, b, c in itertools.product(*map(range, k)))
    out = []
    for mode in (0, 2):
        rt3d.rt3d_debug_set(rt3d.DEBUG_F32_SPLIT, mode)
        try:
            y = lay(x)[..., :cout].double()
        finally:
            rt3d.rt3d_debug_set(rt3d.DEBUG_F32_SPLIT, 1)
        out.append(float((y - ref).norm() / ref.norm()))
    return out + [rt3d.rt3d_last_plan()["kernel"]]


@pytest.mark.parametrize("cout", [32, 64, 96, 128])
@pytest.mark.parametrize("cin,k,density", [(32, (1, 1, 1), 1.0), (64, (1, 1, 1), 1.0), (160, (1, 1, 1), 1.0), (32, (1, 3, 3), 1.0),
                                           (64, (3, 3, 3), 0.4), (64, (3, 3, 3), 1.0)])
def test_no_further_off_than_the_cuda_cores(cout, cin, k, density):
    for x_one_sign in (False, True):
        simt, split, kernel = _errors(cin, cout, k, density, x_one_sign, 0.0)
        assert kernel == 8 and split <= simt, (x_one_sign, simt, split)


@pytest.mark.parametrize("cin,cout,k", [(32, 64, (1, 3, 3)), (64, 128, (3, 3, 3))])
def test_sums_of_one_sign_stay_on_the_cuda_cores(cin, cout, k):
    for w_mean in ("one sign", 1.0, -2.0):
        simt, split, kernel = _errors(cin, cout, k, 1.0, True, w_mean)
        assert kernel == 0 and split == simt
    assert _errors(cin, cout, k, 1.0, True, 0.1)[2] == 8
