"""Rings of the fp32 tensor-core kernel's pipeline: no wait can be answered by an older fill, at any bundle width or count."""
from test_alloc_failures_host import build_and_run


def test_every_wait_is_for_the_next_fill(tmp_path):
    build_and_run(tmp_path, "f32_split_rings")
