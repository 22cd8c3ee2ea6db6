"""An fp32 handle where device memory is short: the layout of the tensor-core kernel is several times as large as that of the CUDA
cores, and a handle or a call for which only the smaller one fits is served by the CUDA cores."""
import pytest
import torch

import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu


def test_layout_of_the_tensor_cores_does_not_fit():
    spec = synth.ConvSpec("m", 512, 512, (3, 3, 3), (1, 1, 1), (1, 1, 1), False)
    L = synth.make_layer(spec, 3, 1, 4, 4, "bernoulli", 0.28)
    lays = [nets.ConvLayer(spec, L["w"], L["bias"], L["mask"], 4, 4, torch.float32) for _ in range(3)]
    x = nets.to_device(synth.make_input(3, (1, 4, 14, 14, 512)), torch.float32)
    y, want = lays[0].alloc_out(x), lays[0](x)
    simt = lays[0](x, algo=rt3d.ALGO_SIMT)
    lays[0](x)
    assert rt3d.rt3d_last_plan()["kernel"] == 8
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rt3d.rt3d_release_kept()                               # blocks of freed handles, which would hold it
    room = torch.cuda.mem_get_info()[0] - (40 << 20)       # 9 MB for each of the two layouts beside it fit, the 50 MB that it comes with do not
    hold = torch.empty(room, dtype=torch.uint8, device="cuda")
    try:
        lays[1].packed.prepare()
        lays[1](x, y)
        assert rt3d.rt3d_last_plan()["kernel"] == 0 and torch.equal(y, simt)
        lays[1].packed.free()
        lays[2](x, y)
        assert rt3d.rt3d_last_plan()["kernel"] == 0 and torch.equal(y, simt)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(lays[2](x), want) and rt3d.rt3d_last_plan()["kernel"] == 8       # with memory again
