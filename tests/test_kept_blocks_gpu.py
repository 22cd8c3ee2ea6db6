"""Device memory kept from freed handles: taking it does not wait for the device, freeing does, and it can be given back."""
import pytest
import torch

import rt3d_synth as synth
import paper_2007_09835_b200 as rt3d
from paper_2007_09835_b200 import binding as B
from paper_2007_09835_b200 import nets

pytestmark = pytest.mark.gpu

SPEC = synth.ConvSpec("l", 256, 512, (3, 3, 3), (1, 1, 1), (1, 1, 1), True)


@pytest.fixture(scope="module")
def weights():
    return synth.make_layer(SPEC, 3, 0, 4, 4, "bernoulli", 0.4)


def layer(L):
    return nets.ConvLayer(SPEC, L["w"], L["bias"], L["mask"], 4, 4, torch.bfloat16)


def busy(stream):
    """About a third of a second of work on a stream that nothing else waits for, and its end."""
    with torch.cuda.stream(stream):
        torch.cuda._sleep(600_000_000)
        end = torch.cuda.Event()
        end.record()
    return end


def test_first_call_into_a_kept_block_does_not_wait_for_the_device(weights):
    x = nets.to_device(synth.make_input(1, (1, 4, 14, 14, 256)))
    side = torch.cuda.Stream()
    with B.concurrent_kernels():                          # plans whose blocks do not wait for one another
        rt3d.rt3d_release_kept()
        first = layer(weights)
        y = first(x)
        torch.cuda.synchronize()
        del first
        again, out = layer(weights), torch.zeros_like(y)
        allocs = rt3d.rt3d_alloc_count()
        end = busy(side)
        again(x, out)
        assert not end.query()                            # the call returned while the other stream was busy
        assert rt3d.rt3d_alloc_count() == allocs          # and its weights went into the kept block
        torch.cuda.synchronize()
        assert torch.equal(out, y)
    assert rt3d.rt3d_last_device_status() == rt3d.OK


def test_free_waits_for_the_kernels_that_use_the_handle(weights):
    x = nets.to_device(synth.make_input(1, (1, 4, 14, 14, 256)))
    side, lay = torch.cuda.Stream(), layer(weights)
    with B.concurrent_kernels():
        want = lay(x)
        y = torch.zeros_like(want)
        torch.cuda.synchronize()
        busy(side)
        with torch.cuda.stream(side):
            lay(x, y)
            end = torch.cuda.Event()
            end.record()
        assert not end.query()
        lay.packed.free()
        assert end.query()
    assert torch.equal(y, want)


def test_kept_blocks_are_given_back(weights):
    lay = layer(weights)
    lay.packed.prepare()
    rt3d.rt3d_release_kept()
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    del lay
    assert torch.cuda.mem_get_info()[0] == held           # kept
    rt3d.rt3d_release_kept()
    assert torch.cuda.mem_get_info()[0] > held


def test_flags_of_a_tail_split_are_clear_before_its_first_launch(weights):
    """The scratch of a tail split is cleared through the default stream; on a stream that does not wait for that one, the call
    has to."""
    x = nets.to_device(synth.make_input(1, (1, 4, 14, 14, 256)))
    want = layer(weights)(x, algo=B.ALGO_UMMA_PAIR)
    plan = rt3d.rt3d_last_plan()
    assert plan["tail_workers"] > 0, plan
    lay, y, side = layer(weights), torch.zeros_like(want), torch.cuda.Stream()
    with B.concurrent_kernels():
        lay(x, y, algo=B.ALGO_UMMA_PAIR)                  # the same weight layout, no tail split
    assert rt3d.rt3d_last_plan()["tail_workers"] == 0 and rt3d.rt3d_last_plan()["kernel"] == plan["kernel"]
    y.zero_()
    torch.cuda.synchronize()
    end = busy(torch.cuda.default_stream())
    with torch.cuda.stream(side):
        lay(x, y, algo=B.ALGO_UMMA_PAIR)
    assert end.query()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    assert rt3d.rt3d_last_device_status() == rt3d.OK


def test_a_captured_tail_split_outlives_a_larger_one(weights):
    """A call of another shape that needs more scratch leaves the scratch of a captured call in place."""
    lay = layer(weights)
    x, big = (nets.to_device(synth.make_input(1, s + (256,))) for s in ((1, 4, 14, 14), (1, 8, 28, 28)))
    y = lay.alloc_out(x)
    want = lay(x, algo=B.ALGO_UMMA_PAIR).clone()
    workers = rt3d.rt3d_last_plan()["tail_workers"]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lay(x, y, algo=B.ALGO_UMMA_PAIR)
    out = lay.alloc_out(big)
    with B.concurrent_kernels():
        lay(big, out, algo=B.ALGO_UMMA_PAIR)              # its weight layout, without a tail split
    allocs = rt3d.rt3d_alloc_count()
    lay(big, out, algo=B.ALGO_UMMA_PAIR)
    assert rt3d.rt3d_last_plan()["tail_workers"] > workers > 0
    assert rt3d.rt3d_alloc_count() == allocs + 2          # partial tiles and flags
    first = out.clone()
    for _ in range(3):
        y.zero_()
        graph.replay()
        assert torch.equal(y, want)
        assert torch.equal(lay(big, out, algo=B.ALGO_UMMA_PAIR), first)
    assert rt3d.rt3d_last_device_status() == rt3d.OK
