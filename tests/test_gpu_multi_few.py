"""Few markers with long vectors, FP4 rows without a K split: rows cut into parts of 4,096 individuals
when no factors are wanted, right at the parts' edges and at the speed of many blocks."""

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


def _panel(n_v, n_f, s, seed):
    rng = np.random.default_rng(seed)
    lo, hi = rng.integers(0, s, size=(2, n_v, (n_f + 15) // 16 * 16), dtype=np.uint8)
    g = (lo | (hi << 4)).astype(np.uint8)
    g[rng.random(g.shape) < 0.02] = 0xFF
    return g


@pytest.mark.parametrize("s", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n_v,n_f", [(2, 4095), (3, 4097), (9, 8192), (2, 12289), (17, 20000), (5, 61441)])
def test_rows_in_parts(s, n_v, n_f):
    """The rows (tallies, JOINT values: both follow from the rows alone) at part edges."""
    g = _panel(n_v, n_f, s, seed=100 * s + n_v)
    et, ec = oracle.ccc2_multi_all(g, n_f, s, norm=1)
    t, c = run_multi(g, n_f, s, norm=1, operand=2, split=1)
    assert_tally_equal(t, et, f"s={s}")
    assert_ccc_close(c, ec, what=f"s={s}")
    t, c = run_multi(g, n_f, s, norm=0, operand=2, split=1)
    assert_tally_equal(t, et, f"s={s}")


def test_preparation_keeps_the_gpu_busy():
    """What a call does besides its tally kernel (the rows' preparation) against writing the rows
    with a fill: reading a byte per entry and writing s / 2 takes less than four times as long (1.1
    measured; 11 with a block per marker)."""
    import torch

    import paper_1705_08213_gb300 as ccc
    n_v, n_f, s, calls = 30, 1000000, 8, 5
    g = to_device_bytes(np.random.default_rng(1).integers(0, 256, (n_v, n_f), dtype=np.uint8))
    opts = ccc.ccc_opts_default(norm=1, operand=2)
    ws = workspace(ccc.ccc_multi_workspace_size(g, n_f, s, opts))
    opts = ccc.ccc_opts_default(norm=1, operand=2, workspace=ws)
    opts.split = 1
    n = ccc.ccc2_count(n_v)
    t = torch.empty(n, s * s, dtype=torch.int32, device="cuda")
    c = torch.empty(n, s * s, dtype=torch.float32, device="cuda")
    rows = torch.empty(ws.numel() // 2, dtype=torch.uint8, device="cuda")  # e2m1: half of the e4m3 rows

    def timed(call):
        best = float("inf")
        for _ in range(5):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            call()
            ccc.ccc_timing_enable()
            ccc.ccc_timing_read()
            start.record()
            for _ in range(calls):
                call()
            end.record()
            end.synchronize()
            best = min(best, (start.elapsed_time(end) - ccc.ccc_timing_read()[0]) / calls)
            ccc.ccc_timing_enable(False)
        return best

    prepare = timed(lambda: ccc.ccc2_multi_tally_metric(g, n_f, s, t, c, opts))
    fill = timed(lambda: rows.fill_(1))
    print(f"preparation {prepare * 1e3:.0f} us, fill of {rows.numel() / 1e6:.0f} MB {fill * 1e3:.0f} us")
    assert prepare < 4 * fill + 0.02, (prepare, fill)
