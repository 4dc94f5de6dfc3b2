"""In the build with checked gathers (MF_CHECK_BOUNDS) the lattice kernels' accesses to arrays in device memory go
through the checking macros of mf_check.cuh, as the list solver's do."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1507_01926_gb300", "csrc")
STATE = re.compile(r"(?:(?<![\w.])L|D\.lat)\.(?:r|ex|d|drain|back|inbox|mask|ret|slots|state|bits)\[(\w*)")
LISTS = re.compile(r"D\.lat\.list\[[^]]*\]\[(\w*)")
PASSED = re.compile(r"(?<![\w.>])(?:drain|mask|ret)\[(?!TV\])(\w*)")  # the same arrays as arguments
GRAPH = re.compile(r"(?<!\w)D\.(?:row|head|cap|rev|out_flow)\[(\w*)")


@pytest.mark.parametrize("name,least", [("mf_lattice.cuh", 30), ("mf_lattice2.cu", 25), ("mf_lattice3.cu", 20)])
def test_every_gather_of_the_lattice_kernels_is_checked(name, least):
    text = open(os.path.join(CSRC, name)).read()
    found = [m for p in (STATE, LISTS, PASSED, GRAPH) for m in p.finditer(text)]
    assert len(found) >= least  # the patterns still match the code
    bare = [text[m.start():text.index("\n", m.start())] for m in found if not m.group(1).startswith("MF_")]
    assert not bare, bare
