"""FP4 operand rows, PERSNP factors and staged outputs of the s-state path against the oracle.

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
from tests.gpu_util import (assert_ccc_close, assert_tally_equal, run_multi, to_device_bytes,
                            workspace)

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


# (s, operand): FP4 and e4m3 (1) tiles; more than eight states are e4m3 by themselves.
@pytest.mark.parametrize("s,operand", [(2, 0), (3, 0), (5, 0), (7, 0), (3, 1), (5, 1), (7, 1),
                                       (9, 0), (10, 0), (11, 0), (13, 0),
                                       (14, 0), (15, 0)])
@pytest.mark.parametrize("dv", [-1, 0, 1])
@pytest.mark.parametrize("norm", [0, 1])
def test_staged_outputs(s, operand, dv, norm):
    """Outputs stored as runs (S = 2 and odd S): nothing outside the pairs of the call."""
    import torch

    import paper_1705_08213_gb300 as ccc
    rng = np.random.default_rng(10 * s + dv + 1)
    n_f, ss = 100, s * s
    n_v = 3 * 8 * (32 // s) + 32 // s + dv  # blocks of 8 PW and 6 PW markers, runs of PW
    npairs = n_v * (n_v - 1) // 2
    lo, hi = rng.integers(0, s + 1, size=(2, n_v, 112), dtype=np.uint8)
    g = (lo | (hi << 4)).astype(np.uint8)
    dev = to_device_bytes(g)
    opts = ccc.ccc_opts_default(norm=norm, operand=operand)
    opts.split = 1
    ws = workspace(ccc.ccc_multi_workspace_size(dev, n_f, s, opts))
    opts = ccc.ccc_opts_default(norm=norm, workspace=ws, operand=operand)
    opts.split = 1
    guard = 64
    inner = slice(guard, guard + npairs * ss)
    t = torch.full((npairs * ss + 2 * guard,), -7, dtype=torch.int32, device="cuda")
    c = torch.full((npairs * ss + 2 * guard,), -7.0, dtype=torch.float32, device="cuda")
    ccc.ccc2_multi_tally_metric(dev, n_f, s, t[inner].view(npairs, ss), c[inner].view(npairs, ss), opts)
    torch.cuda.synchronize()
    assert ccc.ccc_status(opts) == ccc.CCC_OK
    for out in (t, c):
        assert bool((out[:guard] == -7).all()) and bool((out[inner.stop:] == -7).all())
    et, ec = oracle.ccc2_multi_all(g, n_f, s, norm=norm)
    assert_tally_equal(t[inner].view(npairs, ss).cpu().numpy(), et, f"s={s} n_v={n_v}")
    assert_ccc_close(c[inner].view(npairs, ss).cpu().numpy(), ec, what=f"s={s} n_v={n_v}")
