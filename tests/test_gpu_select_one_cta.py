"""Selections that one CTA makes by itself (rows of up to 2048 tokens), with digits taken from the range of the row's keys."""
import numpy as np
import pytest

from test_gpu_parity import _select_case

pytestmark = pytest.mark.gpu


# the ends of the one-CTA range and the first row beyond it
@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 2047, 2048, 2049])
def test_select_ranges_of_keys(oracle, n):
    rng = np.random.default_rng(n)
    base = {"alike": np.full((2, n), 3.25),                                      # no digit at all
            "two": 3.25 + (rng.random((2, n)) < 0.5) * 2.0 ** -20,               # one bit or a few
            "narrow": 1000.0 + rng.integers(0, 4096, (2, n)) * 2.0 ** -10,       # about one digit
            "octaves": np.exp(rng.standard_normal((2, n)) * 2),                  # two digits
            "signs": rng.standard_normal((2, n)) * 1e30}                         # all 32 bits
    base["special"] = base["signs"].copy()
    base["special"][:, ::3] = np.nan
    base["special"][:, 1::5] = np.inf
    base["special"][:, 2::7] = -np.inf
    base["special"][:, 3::11] = -0.0
    for name, s in base.items():
        for k in sorted({0, 1, n // 3, n - 1, n}):
            _select_case(oracle, s.astype(np.float32), k, n_always=3 if name == "two" else 0)


@pytest.mark.parametrize("B", [3, 148, 149, 400])
def test_select_many_rows(oracle, B):
    """Rows on an SM each, and more rows than SMs."""
    rng = np.random.default_rng(B)
    _select_case(oracle, rng.standard_normal((B, 700)).astype(np.float32), 300, n_always=2)
