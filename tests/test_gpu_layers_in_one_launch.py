"""The projections of a block that share one launch (keys and values; with SelectQ&K keys, values and queries)."""
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2506_05096_b200 import binding as A
from helpers import to_dev_bf16
from test_gpu_block import _bits, device_chain, make_block

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_05096_b200", "csrc")


@pytest.fixture(scope="module")
def columns(tmp_path_factory):
    """Columns of a tile and columns that a matrix takes, as the launch chooses them."""
    exe = str(tmp_path_factory.mktemp("tiles") / "tiles")
    main = """#include <cstdio>
              #include <cstdlib>
              #include "linear_tiles.cuh"
              int main(int, char **a) {
                  const int rows = atoi(a[1]), n = atoi(a[2]), mats = atoi(a[3]), bn = astraea::choose_bn(rows, n, mats, atoi(a[4]));
                  printf("%d %d", bn, astraea::mat_columns(n, mats, bn));
              }"""
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-x", "c++", "-", "-o", exe], input=main, text=True, check=True)
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    return lambda rows, D, mats: tuple(int(v) for v in subprocess.check_output([exe, str(rows), str(D), str(mats), str(pairs)]).split())


# padded: columns between the end of each matrix (of two, of three) and the next one's start, 0 with whole halves of a tile
@pytest.mark.parametrize("B,H,d,N,padded", [(1, 8, 72, 1300, (0, 0)), (2, 5, 64, 333, (0, 0)), (1, 1, 64, 257, (0, 0)), (1, 4, 128, 700, (0, 0)),
                                            (2, 16, 72, 1000, (0, 0)),
                                            (3, 5, 64, 1900, (64, 64)), (2, 13, 64, 2000, (32, 32)), (6, 7, 64, 1900, (64, 64)),
                                            (3, 7, 64, 1500, (64, 32)), (6, 8, 72, 1800, (64, 0))])
def test_projections_in_one_launch_equal_single_calls(columns, B, H, d, N, padded):
    """Bit for bit (the contraction of an output does not depend on the tile it is in): the block against its layers as single calls,
    and SelectQ&K against the same layers on the sequence of the selected tokens alone."""
    rng = np.random.default_rng(95)
    D, hidden, N_text = H * d, 128, 9
    assert padded == (columns(B * N, D, 2)[1] - D, columns(B * (N // 2 + 1), D, 3)[1] - D)
    bits, tk_bits, tv_bits = make_block(rng, B, H, d, hidden, N_text)
    Wd = {n: to_dev_bf16(a) for n, a in bits.items()}
    W = A.block_weights(Wd, hidden)
    tk, tv, x, cache = (to_dev_bf16(a) for a in (tk_bits, tv_bits, _bits(rng, B, N, D), _bits(rng, B, N, D)))
    ws = torch.zeros(A.astraea_block_workspace_bytes(B, H, N, d, hidden), dtype=torch.uint8, device="cuda")
    M = N // 2 + 1
    idx = torch.from_numpy(np.stack([np.sort(rng.choice(N, M, replace=False)) for _ in range(B)]).astype(np.int32)).cuda()
    score = torch.empty(B, N, device="cuda")

    def block(flags):
        y, lse = cache.clone(), torch.zeros(B, H, N, device="cuda")
        A.astraea_block_step(x, W, x.clone(), lse, None, y, tk, tv, N_text, score, idx, None, B, H, N, N, d, M,
                             flags=flags | A.BLOCK_REUSE_SELECTION, workspace=ws)
        A.astraea_poll_error(ws)
        return y, lse

    y, lse = block(0)
    y2, lse2 = cache.clone(), torch.zeros(B, H, N, device="cuda")
    device_chain(Wd, x, idx, M, tk, tv, N_text, y2, lse2, B, H, N, d, hidden)
    # (device_chain gives the attention no room to cut keys: at these sizes none are)
    assert torch.equal(y.view(torch.int16), y2.view(torch.int16)) and torch.equal(lse, lse2)
    y, lse = block(A.BLOCK_SELECT_QK)
    rows = idx.long()
    take = lambda t: torch.stack([t[b, rows[b]] for b in range(B)])  # noqa: E731
    y3, lse3 = take(cache), torch.zeros(B, H, M, device="cuda")
    device_chain(Wd, take(x), torch.arange(M, dtype=torch.int32, device="cuda").repeat(B, 1), M, tk, tv, N_text, y3, lse3, B, H, M, d, hidden)
    assert torch.equal(take(y).view(torch.int16), y3.view(torch.int16))
    assert all(torch.equal(lse[b][:, rows[b]], lse3[b]) for b in range(B))
