"""Loops over nodes step without a sign.

A grid may have up to 2^31 - 1 nodes, so a node and the stride after it fit into
32 bits only without a sign: where a launch has a thread a node (the FP64
searches) their sum passes 2^31 on every grid of more than 2^30 nodes, and a
signed index would go on below 0.  From the source: no loop over nodes adds to
a signed index, and on the CPU: the steps of such loops cover every node once.
"""
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_14675_gb300", "csrc")


def test_no_node_loop_adds_to_a_signed_index():
    bad = []
    for name in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"for \((int j\b[^;]*)?;\s*j < [^;]*;\s*j \+= [^)]*\)", src):
            if not (m.group(1) is None and "unsigned j = blockIdx.x" in src):
                bad.append((name, m.group(0)))
        for m in re.finditer(r"\bj \+ stride < (end|n)\b", src):
            if name != "dp_gmres.cu" or "unsigned n = (unsigned)g.n_nodes, stride" not in src:
                bad.append((name, m.group(0)))
    assert not bad, bad


def test_steps_of_a_launch_with_a_thread_a_node():
    # the arithmetic of sweep_kernel and sweep_nodes on 2^31 - 2 nodes (993 x 906 x 217 x 11), blocks of 64
    n = 993 * 906 * 217 * 11
    assert n == 2 ** 31 - 2
    blocks = -(-n // 64)
    stride = np.uint32(blocks * 64)                     # 2^31, which an int holds as -2^31
    assert int(stride.astype(np.int32)) == -2 ** 31
    for j in (0, 1, 2 ** 30, n - 1):
        first = np.uint32(j)
        assert first < np.uint32(n) and not np.uint32((int(first) + int(stride)) % 2 ** 32) < np.uint32(n)
