"""A node's line and mass index from its compact index, on the CPU.

The division by the number of mass nodes is a multiplication.  With 2^40 / n_m as
the factor its product left 64 bits from 2^24 lines (n0 n1 n2) on, and nodes of
such grids came out on other lines, with mass indexes outside the grid.
"""
import subprocess

from test_search64_host import compile_host


def test_every_line_of_every_grid(tmp_path):
    out = subprocess.run([compile_host(tmp_path, "decode_host")], check=True, capture_output=True, text=True).stdout
    looked, wrong = map(int, out.split())
    assert looked > 10 ** 7 and wrong == 0


def test_the_former_factor_left_64_bits():
    # what the test above rests on: 2^24 lines of four nodes, the first node of the last line
    n_m, line = 4, 2 ** 24
    j = line * n_m
    assert j < 2 ** 31 and (j * (2 ** 40 // n_m) % 2 ** 64) >> 40 != line
