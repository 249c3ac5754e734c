"""Bookkeeping of the device-block cache (csrc/devcache.cuh, compiled for the CPU over a
fake allocator with two devices): blocks come back to the device they were allocated
on, whichever is current when they are released."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_blocks_return_to_their_device(tmp_path):
    exe = str(tmp_path / "devcache_check")
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "native", "devcache_check.cu")],
                   check=True, capture_output=True, timeout=300)
    big = 100 << 20
    steps = [
        ("use 0", "cur 0"),
        ("alloc 1 1000", "malloc 0 1024;block 1;cur 0"),
        (f"alloc 2 {big}", f"malloc 0 {big};block 2;cur 0"),
        ("use 1", "cur 1"),
        ("alloc 3 1000", "malloc 1 1024;block 3;cur 1"),
        # a context of device 0 closed while device 1 is current, beside one of device 1
        ("release 1 2 3 -1", "sync 0;sync 1;cur 1"),
        ("alloc 4 1000", "block 3;cur 1"),
        (f"alloc 5 {big}", f"malloc 1 {big};block 4;cur 1"),  # device 0's is not handed out here
        ("use 0", "cur 0"),
        (f"alloc 6 {big}", "block 2;cur 0"),
        ("alloc 7 1010", "block 1;cur 0"),                     # the same rounded size
        ("release 5 -1", "sync 1;cur 0"),
        ("release 6 4 -1", "sync 0;sync 1;cur 0"),
        ("trim", "free 1;free 0;free 1;cur 0"),                # released longest ago first, large before small
        ("release 7 -1", "sync 0;cur 0"),
        ("limit 0", "free 0;cur 0"),
    ]
    out = subprocess.run([exe], input="\n".join(s for s, _ in steps) + "\n", capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stderr
    lines = out.stdout.strip().split("\n")
    assert len(lines) == len(steps)
    for (cmd, want), got in zip(steps, lines):
        assert got.split(" held ")[0] == want, (cmd, got)
    assert lines[-1].endswith("held 0")
