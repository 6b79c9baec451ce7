"""Which pieces the merge kernel of a split head reads: the check it makes on the main kernel's record, on the host."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_17404_b200", "csrc")


@pytest.fixture(scope="module")
def pieces_to_merge(tmp_path_factory):
    d = tmp_path_factory.mktemp("merge_range")
    src, so = d / "m.cpp", d / "m.so"
    src.write_text('#include "piece_range.h"\nextern "C" int f(int a, int b, int n) { return trj::pieces_to_merge(a, b, n); }\n')
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so)).f


def test_records_of_a_finished_launch(pieces_to_merge):
    for first, last, want in [(0, 0, 0), (5, 5, 0), (295, 295, 0), (0, 1, 1), (0, 295, 1), (294, 295, 1)]:
        assert pieces_to_merge(first, last, 296) == want


def test_whatever_memory_holds_stays_inside_the_workspace(pieces_to_merge):
    """A stream whose wait ran out leaves no record: any two words may stand there."""
    r = random.Random(1)
    ends = [-2 ** 31, -1, 0, 1, 295, 296, 297, 0x7f7f7f7f, 2 ** 31 - 1]
    for first, last in [(a, b) for a in ends for b in ends] + [(r.randrange(-2 ** 31, 2 ** 31), r.randrange(-2 ** 31, 2 ** 31)) for _ in range(20000)]:
        if pieces_to_merge(first, last, 296):
            assert 0 <= first < last <= 295


def test_the_merge_kernel_makes_the_check():
    text = open(os.path.join(CSRC, "attn_sm100.cu")).read()
    body = text[text.index("tree_attention_combine_kernel(const AtParams p)"):]
    assert body.index("pieces_to_merge(owners.x, owners.y, p.streams)") < body.index("p.slots")
