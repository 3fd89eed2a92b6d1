"""Host-buffer sessions on a model of the CUDA runtime (tests/session_host.cpp): results under orders that streams and events
allow, steps that fail half way, arguments, and how much is sent for at a time."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2506_05096_b200", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    where = tmp_path_factory.mktemp("session_host")
    for header in ("cuda_runtime.h", "cuda_bf16.h"):                  # the model takes their place
        open(where / header, "w").close()
    exe = str(where / "session_host")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wno-unknown-pragmas", "-I", str(where), "-I", CSRC, "-o", exe, os.path.join(HERE, "session_host.cpp")])
    return exe


def _run(program, *args):
    r = subprocess.run([program] + [str(a) for a in args], stdout=subprocess.PIPE, timeout=120, text=True)
    assert r.returncode == 0, (args, r.stdout)
    return [int(v) for v in r.stdout.split()]


# B, H, d, N_sel, n_always: one chunk; two chunks of rows, the second one shorter; batch elements that go together, all of them, and two and
# one; too many for the path by rows, which go by head groups, one a head and several heads to a group
SHAPES = [(1, 2, 64, 300, 7), (1, 8, 64, 4000, 60), (2, 3, 64, 700, 0), (12, 1, 64, 300, 0), (3, 8, 64, 1100, 1), (13, 2, 64, 300, 3), (13, 14, 72, 40, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("shared", [0, 1])
def test_steps_in_any_order_of_the_streams(program, shape, shared):
    """shared: the output goes back into the buffer that x_cur came from."""
    _run(program, "steps", *shape, shared, 8)


@pytest.mark.parametrize("shape", SHAPES)
def test_unknown_modes_are_refused_before_anything_is_sent_for(program, shape):
    _run(program, "modes", *shape)


# the first step of a session, a later dense one and a sparse one behind them
@pytest.mark.parametrize("k_keep,first", [(100, 1), (100, 0), (40, 0)])
@pytest.mark.parametrize("shape", [(1, 2, 64, 100, 7), (3, 2, 64, 100, 0), (13, 2, 64, 100, 3)])
def test_a_step_that_fails_leaves_nothing_under_way(program, shape, k_keep, first):
    """Whichever call of the step fails: the caller may free its buffers when it gets the error."""
    _run(program, "fail", *shape, k_keep, first)


@pytest.mark.parametrize("shape", SHAPES)
def test_no_copy_in_waits_for_a_copy_back(program, shape):
    """With pageable buffers a copy back holds up the call until it is over, so that whatever is sent for behind it comes late."""
    copies_in, copies_back, late = _run(program, "steps", *shape, 0, 1)[:3]
    assert copies_in > 0 and copies_back > 0 and late == 0


def test_small_batch_elements_share_their_copies(program):
    """No more copies than by head groups (x_cur, and q, k and v of each of up to twelve groups)."""
    for B, H, N in ((2, 1, 300), (5, 2, 300), (12, 1, 300), (12, 4, 100)):
        copies_in, _, _, *ctas = _run(program, "steps", B, H, 64, N, 0, 0, 3)
        assert copies_in <= 3 * H + 1 and sum(ctas) == B * H * ((N + 255) // 256)


def test_chunks_of_a_long_sequence_of_few_heads_fill_the_chip(program):
    """126 CTAs of 250 key tiles: cut so that the two launches that run at a time leave no more than a third of the 148 SMs idle."""
    ctas = _run(program, "steps", 1, 2, 128, 15900, 0, 0, 1)[3:]
    assert all(2 * c > 98 for c in ctas), ctas
