"""Feedback and closed loop without page-locked memory: the buffer's owner, on the CPU against a fake allocator.

Calls for more than 819 states keep their states in page-locked memory of the
grid; where the host has none left they have to take the device buffer
instead of failing.
"""
import os
import re
import subprocess

from test_search64_host import CSRC, compile_host


def test_a_refused_buffer_leaves_no_error_and_keeps_the_old_one(tmp_path):
    r = subprocess.run([compile_host(tmp_path, "pinned_host")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_the_call_takes_the_device_buffer_then(tmp_path):
    src = open(os.path.join(CSRC, "dp_api.cu")).read()
    body = src[src.index("int loop_common("):]
    body = body[:body.index("\n}\n")]
    assert re.search(r"const bool pinned = d_buf != nullptr;", body)
    assert not re.search(r"CK\(cudaMallocHost", body)
