"""The copying warp of the attention kernel (csrc/copy_rows.cuh) on the host, lane by lane: what it copies, and how it leaves
when a wait of its CTA runs out, which no GPU test may bring about."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2506_05096_b200", "csrc")


@pytest.fixture(scope="module", params=[2, 3])
def program(request, tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("copy_rows") / ("stages%d" % request.param))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-Wno-unknown-pragmas", "-DSTAGES=%d" % request.param, "-I", CSRC, "-o", exe,
                           os.path.join(HERE, "copy_rows_host.cpp")])
    return exe


# rows of one 16-byte piece, of several to a batch, of exactly a stage, of more than one stage with a ragged last piece
@pytest.mark.parametrize("rows,tokens,bytes_", [(1, 5, 16), (70, 200, 256), (33, 40, 432), (9, 9, 4096), (7, 30, 4224), (5, 11, 6144)])
def test_copies_the_listed_rows(program, rows, tokens, bytes_):
    for blocks in (1, 3):
        subprocess.run([program, str(rows), str(tokens), str(bytes_), str(blocks), "-1"], check=True, timeout=60)


@pytest.mark.parametrize("give_up", [0, 1, 4])
@pytest.mark.parametrize("rows,bytes_", [(200, 256), (12, 6144)])
def test_a_wait_that_runs_out_parts_no_lanes_and_leaves_no_load_in_flight(program, rows, bytes_, give_up):
    subprocess.run([program, str(rows), "300", str(bytes_), "1", str(give_up)], check=True, timeout=60)
