"""Out of host memory inside a C entry point: a status, on any thread, and never the end of the process.  The blocks kept from
freed handles: bounded, given back, one owner each."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_09835_b200", "csrc")


def build_and_run(tmp_path, name, *more):
    exe = str(tmp_path / name)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", exe,
                           os.path.join(ROOT, "tests", name + ".cpp"), *more])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), (r.returncode, r.stdout[-500:], r.stderr[-500:])


def test_every_allocation_of_the_packers_may_fail(tmp_path):
    build_and_run(tmp_path, "alloc_failures", os.path.join(CSRC, "pack.cpp"))


def test_kept_blocks(tmp_path):
    build_and_run(tmp_path, "kept_blocks")
