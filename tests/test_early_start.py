"""Kernels that may become resident before the one ahead of them has finished (launch_after) read nothing early.

A load through a `const ... __restrict__` pointer counts as read-only for the
compiler, which may move it ahead of the wait.  From the source: control blocks
are never such pointers, and a kernel takes such pointers at all only if it
begins with a test of a volatile flag, behind which no load can be run early.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_14675_gb300", "csrc")


def _kernels():
    for name in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"\n(\w+_kernel)\(([^{}]*)\)\s*\{(.*?)\n\}", src, flags=re.S):
            if "wait_for_previous();" in m.group(3):
                yield m.groups()


KERNELS = list(_kernels())


def test_the_kernels_are_found():
    launched = set()
    for name in os.listdir(CSRC):
        launched |= set(re.findall(r"auto kern = (\w+_kernel)<", open(os.path.join(CSRC, name)).read()))
    assert {"sweep_kernel", "gm_start_kernel", "gm_matvec_kernel", "gm_dots_kernel", "gm_update_kernel",
            "gm_apply_kernel"} == {k for k, _, _ in KERNELS} <= launched


@pytest.mark.parametrize("name,params,body", KERNELS, ids=[k for k, _, _ in KERNELS])
def test_no_load_can_be_moved_ahead_of_the_wait(name, params, body):
    order = re.sub(r"\s+", " ", body).strip()
    order = re.sub(r"^constexpr [^;]*;", "", order).strip()
    assert order.startswith("let_next_start(); wait_for_previous();")
    behind = order[len("let_next_start(); wait_for_previous();"):].strip()
    params = [p.strip() for p in params.split(",")]
    assert not any(re.search(r"\b(GmCtl|Ctl)\s*\*\s*__restrict__", p) and "const" in p for p in params)
    assert not any(re.search(r"\bGmCtl\s*\*\s*__restrict__", p) for p in params)
    if not re.match(r"if \(\*\((const )?volatile int\*\)&\w+->(stop|done)\) return;", behind):
        assert not any("const" in p and "*" in p and "__restrict__" in p for p in params)
