"""Rules that the CUDA sources keep and that no run can show broken at will:
they are read from the source text, without a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1701_06254_gb300", "csrc")


def _source(name):
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", " ", s, flags=re.S)


def test_a_solve_reads_the_error_word_it_gave_to_the_network():
    """A network serves several simulators: the word that a kernel of one
    solve's prediction sets is that solve's own, and it is the one the solve
    reads after its synchronisation."""
    s = _source("sim.cu")
    body = s[s.index("static int s_solve("):]
    given = re.search(r"ws_predict\([^;]*ls->errw_dev \+ (\d+)", body)
    read = re.search(r"ws_check\(ls->errw \+ (\d+)\)", body)
    assert given and read and given.group(1) == read.group(1) != "0"


# What a kernel may declare __restrict__ although it starts while the kernels
# before it still run: data fixed between setups (patterns, matrix values,
# level operators, inverse diagonals, the coarsest inverse).
FIXED = {"rp", "ci", "val", "vh", "vl", "v", "dinv", "invT"}


def _kernels(src):
    """(parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__", src):
        j = src.index("{", m.start())
        if ";" in src[m.start():j]:
            continue
        depth, k = 0, j
        while True:
            depth += {"{": 1, "}": -1}.get(src[k], 0)
            if depth == 0:
                break
            k += 1
        yield src[m.start():j], src[j:k]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_programmatic_kernels_restrict_fixed_data_only(name):
    """A const __restrict__ pointer lets the compiler use read-only loads and
    move them above the wait for the kernel that writes the data."""
    for head, body in _kernels(_source(name)):
        if "pdl_wait" in body:
            names = set(re.findall(r"\*\s*__restrict__\s*(\w+)", head))
            assert names <= FIXED, (" ".join(head.split())[:120], names - FIXED)


def test_lane_numbers_of_wide_rows_are_unsigned():
    """32 lanes per row: the thread's number would pass 2^31 at 2^26 rows, not
    far above the 50M cells that are accepted; as an int it would then name a
    negative row."""
    s = _source("amg.cu")
    m = re.search(r"void tpos_row\((\w+) g,", s)
    assert m and m.group(1) == "unsigned"
