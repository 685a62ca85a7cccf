"""GPU 2-way output by 128-byte lines: arrays at every multiple of 16 bytes, sizes at the edges of
lines (8 pairs), half tiles (64 SNPs) and tiles (128), row ranges; nothing written around them."""

import pytest

import oracle
import synth
from tests.gpu_util import assert_ccc_close, assert_tally_equal, to_device, workspace

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


def _at(count, offset, dtype):
    """(whole buffer, view of count 16-byte records that starts offset records into it)."""
    import torch
    buf = torch.full((count + 16, 4), -7, dtype=dtype, device="cuda")
    return buf, buf[offset:offset + count]


@pytest.mark.parametrize("operand", [1, 2])
@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("n_v,off_t,off_c", [(2, 0, 0), (9, 1, 1), (64, 7, 7), (65, 3, 4), (66, 5, 0),
                                             (128, 2, 6), (129, 6, 6), (193, 4, 3), (257, 1, 7)])
def test_arrays_at_any_record(n_v, off_t, off_c, norm, operand):
    import torch

    import paper_1705_08213_gb300 as ccc
    n_f = 70
    geno = synth.panel_hwe(n_v, n_f, seed=91 + n_v, p_missing=0.05)
    et, ec = oracle.ccc2_all(geno, n_f, norm=norm)
    g = to_device(geno)
    opts = ccc.ccc_opts_default(norm=norm, operand=operand)
    ws = workspace(ccc.ccc_workspace_size(g, n_f, opts, ccc.CCC_OP_2WAY))
    opts = ccc.ccc_opts_default(norm=norm, operand=operand, workspace=ws)
    for i0, i1 in ((0, n_v), (1, n_v), (n_v // 2, n_v - 1)):
        lo, cnt = ccc.ccc2_rows_count(n_v, 0, i0), ccc.ccc2_rows_count(n_v, i0, i1)
        if cnt == 0:
            continue
        tb, t = _at(cnt, off_t, torch.int32)
        cb, c = _at(cnt, off_c, torch.float32)
        ccc.ccc2_tally_metric_rows(g, n_f, i0, i1, t, c, opts)
        assert ccc.ccc_status(opts) == ccc.CCC_OK
        assert_tally_equal(t.cpu().numpy(), et[lo:lo + cnt], f"rows {i0}..{i1}")
        assert_ccc_close(c.cpu().numpy(), ec[lo:lo + cnt], what=f"rows {i0}..{i1}")
        for buf, off in ((tb, off_t), (cb, off_c)):
            assert bool((buf[:off] == -7).all()) and bool((buf[off + cnt:] == -7).all())
