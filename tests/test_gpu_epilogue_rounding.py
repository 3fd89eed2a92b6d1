"""The roundings of the linear layers' epilogue, which the outputs of stacked blocks follow bit for bit."""
import pytest
import torch

from paper_2506_05096_b200 import binding as A

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("listed,compact_res,inplace", [(False, False, False), (True, False, False), (True, True, False), (True, False, True)])
def test_gate_is_rounded_before_the_residual_is_added(listed, compact_res, inplace):
    """Whole numbers below 2^24 make the contraction exact, so that the result is bf16(fl32(fl32(gate * (x W^T + bias)) + residual)) to the
    bit; a residual that all but cancels the product shows a product that was not rounded (one FMA) in most elements."""
    g = torch.Generator("cuda").manual_seed(1)
    B, N, K, N_out = 2, 300, 128, 200
    whole = lambda *s, hi: torch.randint(-hi, hi + 1, s, device="cuda", generator=g).float()  # noqa: E731
    x, w, bias = whole(B, N, K, hi=255), whole(N_out, K, hi=255), whole(N_out, hi=255)
    gate = torch.randn(B, N_out, device="cuda", generator=g).bfloat16()
    f = (x.double() @ w.double().T + bias.double()).float()
    assert f.abs().max() < 2 ** 24
    M = 151 if listed else N
    idx = torch.stack([torch.randperm(N, device="cuda", generator=g)[:M].sort().values for _ in range(B)]).int() if listed else None
    product = gate.float()[:, None] * f
    res = (-product).bfloat16()
    want = (product + res.float()).bfloat16()
    rows = [idx[b].long() if listed else slice(None) for b in range(B)]
    r = torch.stack([res[b, rows[b]] for b in range(B)]) if compact_res else res
    y = res.clone() if inplace else torch.zeros_like(res)
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    A.astraea_gathered_linear_residual(x.bfloat16(), idx, M, w.bfloat16(), bias.bfloat16(), y if inplace else r, gate, y, B, N, K, N_out,
                                       flags=A.LINEAR_COMPACT_RES if compact_res else 0, workspace=ws)
    A.astraea_poll_error(ws)
    for b in range(B):
        assert torch.equal(y[b, rows[b]], want[b, rows[b]])


def test_gelu_next_to_rounding_boundaries():
    """Arguments x + bias whose GELU lies so close to the middle of two bf16 that the place of one fp32 rounding decides."""
    points = [(-0.12451171875, -3.3125, -0.001007080078125), (-0.00142669677734375, -3.609375, -0.00054931640625),
              (-0.00083160400390625, -2.203125, -0.0303955078125), (-0.0023040771484375, -1.9609375, -0.048828125),
              (0.00543212890625, -2.59375, -0.012451171875), (-0.01019287109375, -2.578125, -0.012451171875),
              (0.0030670166015625, -4.03125, -0.00011301040649414062)]
    x, bias, want = (torch.tensor(c, device="cuda").bfloat16() for c in zip(*points))
    n = len(points)
    a, b, y = torch.zeros(1, n, 64, device="cuda").bfloat16(), torch.zeros(64, device="cuda").bfloat16(), torch.zeros(1, n, 64, device="cuda").bfloat16()
    a[0, range(n), range(n)], b[:n] = x, bias
    A.astraea_gathered_linear(a, None, n, torch.eye(64, device="cuda").bfloat16(), b, y, 1, n, 64, 64, flags=A.LINEAR_GELU,
                              workspace=torch.zeros(256, dtype=torch.uint8, device="cuda"))
    assert torch.equal(y[0, range(n), range(n)], want)
