"""Layer norms whose modulation vectors are held in registers, read per row, or only one of them given."""
import numpy as np
import pytest
import torch

from paper_2506_05096_b200 import binding as A
from helpers import bf16_dev_to_f64, f64, to_dev_bf16
from test_gpu_block import _bits

pytestmark = pytest.mark.gpu


# every width of the register arrays with a ragged last vector, rows for less than a warp each (held) and for several (read per row)
@pytest.mark.parametrize("D", [504, 1016, 1152, 1528, 2040, 3064, 4088])
@pytest.mark.parametrize("B,N", [(1, 5), (3, 77), (2, 4000)])
def test_layernorm_forms(oracle, D, B, N):
    """Against the oracle on sampled rows: one rounding to bf16 (2^-9 relative) of results of order 1 to 10."""
    rng = np.random.default_rng(D + N)
    x, s, t = _bits(rng, B, N, D), _bits(rng, B, D, scale=0.3), _bits(rng, B, D, scale=0.3)
    rows = np.unique(np.concatenate([[0, N - 1], rng.integers(0, N, 6)]))
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    for sc, sh in ((s, t), (s, None), (None, t), (None, None)):
        y = torch.zeros(B, N, D, dtype=torch.bfloat16, device="cuda")
        A.astraea_layernorm_modulate(to_dev_bf16(x), None, N, None if sc is None else to_dev_bf16(sc), None if sh is None else to_dev_bf16(sh), y, B, N, D,
                                     workspace=ws)
        A.astraea_poll_error(ws)
        xr = f64(x)[:, rows]
        want = (xr - xr.mean(2, keepdims=True)) / np.sqrt(xr.var(2, keepdims=True) + 1e-6)
        if sc is not None:
            want = want * (1.0 + f64(sc)[:, None])
        if sh is not None:
            want = want + f64(sh)[:, None]
        got = bf16_dev_to_f64(y)[:, rows]
        assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-4).all()
        assert bool((y != 0).any(2).all())                          # every row was written


# per width: blocks of an SM in the form that holds the vectors, and rows a warp just below and just above the lines of the launch rule
@pytest.mark.parametrize("D,blocks,loads", [(504, 8, (1.0, 1.04)), (1016, 5, (1.15, 1.4, 1.7)), (1152, 5, (1.15, 1.35, 1.5)), (1528, 4, (1.15, 1.3)),
                                            (2040, 3, (1.35, 1.5)), (3064, 3, (1.0, 1.04)), (4088, 2, (1.08, 1.2))])
def test_layernorm_second_row_of_a_warp_in_another_batch_element(D, blocks, loads):
    """Two batch elements of which some warps have a row each, so that held vectors must be fetched anew; all rows, against 64 bits."""
    warps = torch.cuda.get_device_properties(0).multi_processor_count * blocks * 4
    g = torch.Generator("cuda").manual_seed(D)
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    for load in loads:
        N = int(warps * load) // 2
        x, s, t = (torch.randn(2, *n, device="cuda", generator=g).bfloat16() for n in ((N, D), (D,), (D,)))
        y = torch.zeros(2, N, D, dtype=torch.bfloat16, device="cuda")
        A.astraea_layernorm_modulate(x, None, N, s, t, y, 2, N, D, workspace=ws)
        A.astraea_poll_error(ws)
        x = x.double()
        want = (x - x.mean(2, keepdim=True)) * torch.rsqrt(x.var(2, unbiased=False, keepdim=True) + 1e-6) * (1.0 + s.double()[:, None]) + t.double()[:, None]
        assert bool(((y.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-4).all())       # one rounding to bf16 (2^-9), fp32 before it
