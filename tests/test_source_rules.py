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
