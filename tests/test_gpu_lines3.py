"""GPU 3-way output by 128-byte lines (genotype-class tiles of 128 x 120 and 128 x 128 SNPs): arrays at
every multiple of 16 bytes, sizes at the edges of lines (4 triples), half tiles and tiles, slab
ranges, panels without missing entries and with more than the compacted rows take."""

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
    """(whole buffer, view of count 32-byte records that starts offset 16-byte units into it)."""
    import torch
    buf = torch.full((8 * count + 128,), -7, dtype=dtype, device="cuda")
    return buf, buf[4 * offset:4 * offset + 8 * count].view(count, 8)


@pytest.mark.parametrize("operand", [1, 2])
@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("n_v,n_f,missing,off_t,off_c", [
    (3, 40, 0.1, 0, 0), (6, 300, 0.0, 1, 0), (66, 130, 0.02, 2, 7), (123, 257, 0.3, 3, 4),
    (132, 600, 0.6, 5, 6), (140, 90, 0.05, 4, 1)])
def test_arrays_at_any_16_bytes(n_v, n_f, missing, off_t, off_c, norm, operand):
    import torch

    import paper_1705_08213_gb300 as ccc
    geno = synth.panel_hwe(n_v, n_f, seed=17 + n_v, p_missing=missing)
    g = to_device(geno)
    opts = ccc.ccc_opts_default(norm=norm, operand=operand)
    ws = workspace(ccc.ccc_workspace_size(g, n_f, opts, ccc.CCC_OP_3WAY))
    opts = ccc.ccc_opts_default(norm=norm, operand=operand, workspace=ws)
    et, ec = oracle.ccc3_slabs(geno, n_f, norm=norm)
    for j0, j1 in ((0, n_v), (n_v // 3, n_v - n_v // 4)):
        lo, cnt = ccc.ccc3_count(n_v, 0, j0), ccc.ccc3_count(n_v, j0, j1)
        if cnt == 0:
            continue
        tb, t = _at(cnt, off_t, torch.int32)
        cb, c = _at(cnt, off_c, torch.float32)
        ccc.ccc3_tally_metric(g, n_f, j0, j1, t, c, opts)
        assert ccc.ccc_status(opts) == ccc.CCC_OK
        assert_tally_equal(t.cpu().numpy(), et[lo:lo + cnt], f"slabs {j0}..{j1}")
        assert_ccc_close(c.cpu().numpy(), ec[lo:lo + cnt], what=f"slabs {j0}..{j1}")
        for buf, off in ((tb, off_t), (cb, off_c)):
            end = 4 * off + 8 * cnt
            assert bool((buf[:4 * off] == -7).all()) and bool((buf[end:] == -7).all())
        only = torch.full((cnt, 8), -7, dtype=torch.int32, device="cuda")
        ccc.ccc3_tally(g, n_f, j0, j1, only, opts)
        assert torch.equal(only, t)


@pytest.mark.parametrize("operand", [1, 2])
@pytest.mark.parametrize("n_v,n_f", [(19, 600), (37, 2050), (18, 16383)])
def test_missing_counts_at_the_edges_of_the_lists(n_v, n_f, operand):
    """Middle SNPs with exactly 0, 1, 127 .. 129, 255 .. 257 and more missing entries: the compacted
    rows' two halves, their capacity, and the masked rows that take over beyond it."""
    import numpy as np
    import torch

    import paper_1705_08213_gb300 as ccc
    geno = synth.panel_hwe(n_v, n_f, seed=5 * n_v, p_missing=0.0, pad_seed=2)
    rng = np.random.default_rng(n_v)
    for j in range(n_v):
        for q in rng.choice(n_f, (0, 1, 127, 128, 129, 255, 256, 257, n_f // 2)[j % 9], replace=False):
            w, b = divmod(int(q), 32)
            geno[j, w] = (geno[j, w] & ~(np.uint64(3) << np.uint64(2 * b))) | (np.uint64(2) << np.uint64(2 * b))
    g = to_device(geno)
    opts = ccc.ccc_opts_default(operand=operand)
    ws = workspace(ccc.ccc_workspace_size(g, n_f, opts, ccc.CCC_OP_3WAY))
    opts = ccc.ccc_opts_default(operand=operand, workspace=ws)
    count = ccc.ccc3_count(n_v, 0, n_v)
    t = torch.full((count, 8), -7, dtype=torch.int32, device="cuda")
    c = torch.full((count, 8), -7.0, dtype=torch.float32, device="cuda")
    ccc.ccc3_tally_metric(g, n_f, 0, n_v, t, c, opts)
    assert ccc.ccc_status(opts) == ccc.CCC_OK
    et, ec = oracle.ccc3_slabs(geno, n_f)
    assert_tally_equal(t.cpu().numpy(), et)
    assert_ccc_close(c.cpu().numpy(), ec)
