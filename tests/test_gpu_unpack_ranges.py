"""GPU K-block-major unpack: K ranges of at least four K blocks (of 256 e2m1 or 128 e4m3 entries), with
row ends inside the first and the last block of a range, with and without the factors."""

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
@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("n_v,n_f", [(9, 300), (33, 769), (20, 1024), (20, 1025), (20, 1281), (50, 2047),
                                     (50, 2049), (300, 2305), (130, 9000)])
def test_ranges(n_v, n_f, norm, operand):
    geno = synth.panel_hwe(n_v, n_f, seed=3 * n_v + n_f, p_missing=0.03, pad_seed=4)
    et, ec = oracle.ccc2_all(geno, n_f, norm=norm)
    t, c = run_2way(geno, n_f, path=0, split=2, norm=norm, operand=operand)
    assert_tally_equal(t, et)
    assert_ccc_close(c, ec)
