"""GPU operand unpack at its edges: rows that end inside a word, a K stage or one thread's two words
(8,192 entries: the line between the fused and the two-kernel form for few SNPs), the K-block-major form's
four-block groups, with arbitrary bits past n_f."""

import pytest

import oracle
import synth
from tests.gpu_util import assert_ccc_close, assert_tally_equal, run_2way

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


@pytest.mark.parametrize("operand", [1, 2])
@pytest.mark.parametrize("n_v,n_f,split", [
    (5, 1, 1), (17, 31, 1), (17, 33, 1), (20, 255, 1), (20, 4097, 1), (33, 8191, 1), (33, 8192, 1),
    (33, 8193, 1), (1300, 300, 1), (20, 1023, 2), (20, 1025, 3), (40, 8193, 5)])
def test_edges(n_v, n_f, split, operand):
    geno = synth.panel_hwe(n_v, n_f, seed=n_v + n_f, p_missing=0.03, pad_seed=9)
    et, ec = oracle.ccc2_all(geno, n_f)
    t, c = run_2way(geno, n_f, path=0, split=split, operand=operand)
    assert_tally_equal(t, et)
    assert_ccc_close(c, ec)
