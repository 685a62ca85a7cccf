"""FP4 operand rows and PERSNP factors of the s-state path against the oracle.

The rows and the factors come from one read of a marker's bytes.  Every byte
value occurs (codes at and past s make the individual missing, also in one half
only), the bytes past the last individual are no genotypes, and the sizes cover
individual counts around 8 entries (one packed word), 16 bytes (the second half
of a thread's load), 32 (a thread) and 4,096 (a block's step), and marker counts
around the 8 PW of an operand row block.
"""

import numpy as np
import pytest

import oracle
from tests.gpu_util import assert_ccc_close, assert_tally_equal, run_multi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


@pytest.mark.parametrize("s", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n_f", [1, 9, 16, 17, 31, 33, 4096, 4127])
def test_rows_and_factors(s, n_f):
    rng = np.random.default_rng(1000 * s + n_f)
    n_v = 8 * (32 // s) + 1 + s % 2
    ld = (n_f + 15) // 16 * 16
    g = rng.integers(0, 256, size=(n_v, ld), dtype=np.uint8)
    # Half of the entries are genotypes (both codes below s), so that pairs share individuals.
    lo, hi = rng.integers(0, s, size=(2, n_v, ld), dtype=np.uint8)
    g = np.where(rng.random((n_v, ld)) < 0.5, lo | (hi << 4), g).astype(np.uint8)
    g[1, :] = 0xFF  # a marker without genotypes
    for norm in (0, 1):
        t, c = run_multi(g, n_f, s, norm=norm, split=1)
        et, ec = oracle.ccc2_multi_all(g, n_f, s, norm=norm)
        assert_tally_equal(t, et, f"s={s} n_f={n_f}")
        assert_ccc_close(c, ec, what=f"s={s} n_f={n_f}")
