"""The greedy rule's orientation sets (sbmt_greedy.cuh), compiled for the host:
each word of them has one writer, so that what a pair's two entries and its
undecided set hold comes from one evaluation of the filter."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_19474_gb300", "csrc")


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda = next((d for d in (os.environ.get("CUDA_HOME"), "/usr/local/cuda") if d and os.path.isdir(d)), None)
    if cxx is None or cuda is None:
        pytest.skip("no host compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("greedy") / "greedy_sets")
    subprocess.run([cxx, "-O1", "-std=c++17", "-w", "-ffp-contract=off", "-I", CSRC, "-I", os.path.join(cuda, "include"),
                    "-o", exe, os.path.join(HERE, "greedy_sets.cpp")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return {int(l.split()[0]): [int(x) for x in l.split()[1:]] for l in out.splitlines()}


@pytest.mark.parametrize("G", [8, 16, 32])
def test_one_writer_a_pair(rows, G):
    """Cells with a vertex at the edge of the band of a pair half the cycle apart,
    which the determinants from the pair's two ends decide differently: the sets do
    not depend on the order in which the lanes run, and every sign read from them is
    the exact one."""
    cells, order, sign = rows[G]
    assert cells >= 100
    assert order == 0, "%d of %d cells: sets depend on the lanes' order" % (order, cells)
    assert sign == 0
