"""GPU popcount path at the edges of its tiles (32 SNPs), of the four-word groups of its carry-save
adders (256 entries) and of its stages (512), with and without a K split, and all-ones panels,
where every running word overflows."""

import numpy as np
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


@pytest.mark.parametrize("split", [1, 3])
@pytest.mark.parametrize("n_v,n_f", [(2, 1), (31, 64), (32, 65), (33, 255), (34, 257), (64, 511),
                                     (65, 513), (66, 1025), (97, 1537)])
def test_edges(n_v, n_f, split):
    geno = synth.panel_hwe(n_v, n_f, seed=31 * n_v + n_f, p_missing=0.05, pad_seed=3)
    t, c = run_2way(geno, n_f, path=1, split=split)
    et, ec = oracle.ccc2_all(geno, n_f)
    assert_tally_equal(t, et)
    assert_ccc_close(c, ec)


@pytest.mark.parametrize("word", [0x0000000000000000, 0x5555555555555555, 0xFFFFFFFFFFFFFFFF])
def test_constant_panels(word):
    n_v, n_f = 35, 32 * 80
    geno = np.full((n_v, 80), word, dtype=np.uint64)
    t, c = run_2way(geno, n_f, path=1)
    et, ec = oracle.ccc2_all(geno, n_f)
    assert_tally_equal(t, et)
    assert_ccc_close(c, ec)
