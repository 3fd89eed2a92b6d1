"""The projections of a block that share one launch (keys and values; with SelectQ&K keys, values and queries)."""
import numpy as np
import pytest
import torch

from paper_2506_05096_b200 import binding as A
from helpers import to_dev_bf16
from test_gpu_block import _bits, device_chain, make_block

pytestmark = pytest.mark.gpu


# widths whose halves of a tile leave a remainder in every matrix, an odd number of halves in all, less than half a tile, whole tiles
@pytest.mark.parametrize("B,H,d,N", [(1, 8, 72, 1300), (2, 5, 64, 333), (1, 1, 64, 257), (1, 4, 128, 700), (2, 16, 72, 1000)])
def test_projections_in_one_launch_equal_single_calls(B, H, d, N):
    """Bit for bit (the contraction of an output does not depend on the tile it is in): the block against its layers as single calls,
    and SelectQ&K against the same layers on the sequence of the selected tokens alone."""
    rng = np.random.default_rng(95)
    D, hidden, N_text = H * d, 128, 9
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
