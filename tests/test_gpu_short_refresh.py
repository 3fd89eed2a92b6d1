"""Refreshes of the reference inputs by CTAs that the attention leaves idle."""
import pytest
import torch

from paper_2506_05096_b200 import binding as A

pytestmark = pytest.mark.gpu


# rows of one lane's width and odd widths; one unit, several units with a remainder; more rows than idle CTAs' passes; a batch
@pytest.mark.parametrize("B,H,d,N_v,N_t,k", [(1, 2, 64, 256, 0, 128), (2, 3, 72, 200, 7, 77), (1, 3, 128, 700, 0, 699), (2, 24, 64, 300, 5, 300), (1, 9, 72, 2000, 8, 555)])
def test_refresh_beside_a_short_attention(B, H, d, N_v, N_t, k):
    """Bit for bit: listed rows are the current inputs, the others what they were."""
    N, D, M = N_v + N_t, H * d, k + N_t
    g = torch.Generator("cuda").manual_seed(4)
    x, x_ref, q, kk, v, out = (torch.randn(B, N, D, dtype=torch.bfloat16, device="cuda", generator=g) for _ in range(6))
    lse, n_skip, score = torch.zeros(B, H, N, device="cuda"), torch.zeros(B, N_v, dtype=torch.int32, device="cuda"), torch.empty(B, N_v, device="cuda")
    sel, rem = torch.empty(B, M, dtype=torch.int32, device="cuda"), torch.empty(B, N_v - k, dtype=torch.int32, device="cuda")
    ws = A.new_workspace(A.OP_STEP, B, H, N, M, d)
    want = x_ref.clone()
    A.astraea_step(x, x_ref, lse, n_skip, q, kk, v, out, score, sel, rem, B, H, N, N_v, d, k, workspace=ws)
    A.astraea_poll_error(ws)
    for b in range(B):
        want[b, sel[b].long()] = x[b, sel[b].long()]
    assert torch.equal(x_ref.view(torch.int16), want.view(torch.int16))
