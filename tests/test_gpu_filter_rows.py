"""GPU thresholded 2-way output (FP4 tiles of 128 x 120 SNPs): the row-wise first test must let every
hit through at any share of missing entries (its bound on n_ij is loosest where many are missing),
any threshold, a SNP whose factor is zero (gamma 1, one allele only), an all-missing SNP and tile edges."""

import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import CCC_RTOL, to_device, workspace

pytestmark = pytest.mark.gpu

HIT = np.dtype([("i", np.int32), ("j", np.int32), ("tally", np.int32, 4), ("ccc", np.float32, 4)])


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


@pytest.mark.parametrize("gamma", [2.0 / 3.0, 1.0])
@pytest.mark.parametrize("threshold", [-0.01, 0.0, 0.02, 0.1, 0.15])
@pytest.mark.parametrize("n_v,n_f,missing", [(119, 300, 0.0), (121, 515, 0.02), (128, 256, 0.3),
                                             (241, 300, 0.7), (130, 40, 0.95)])
def test_hits_equal_the_oracle(n_v, n_f, missing, threshold, gamma):
    import torch

    import paper_1705_08213_gb300 as ccc
    geno = synth.panel_hwe(n_v, n_f, seed=7 * n_v, p_missing=missing, pad_seed=5)
    geno[3] = np.uint64(0)                   # allele 0 only
    geno[n_v - 2] = np.uint64(0xFFFFFFFFFFFFFFFF)  # allele 1 only
    geno[n_v // 2] = np.uint64(0xAAAAAAAAAAAAAAAA)  # all missing
    geno[n_v - 1] = geno[0]
    t, c = oracle.ccc2_all(geno, n_f, gamma=gamma)
    mx = c.max(1)
    tie = np.abs(mx - threshold) <= CCC_RTOL * abs(threshold)
    g = to_device(geno)
    opts = ccc.ccc_opts_default(gamma=gamma, operand=ccc.CCC_OPERAND_E2M1)
    ws = workspace(ccc.ccc_workspace_size(g, n_f, opts, ccc.CCC_OP_2WAY))
    opts = ccc.ccc_opts_default(gamma=gamma, operand=ccc.CCC_OPERAND_E2M1, workspace=ws)
    cap = len(mx)
    hits = torch.zeros(cap * HIT.itemsize, dtype=torch.uint8, device="cuda")
    n_hits = torch.zeros(1, dtype=torch.int64, device="cuda")
    ccc.ccc2_filter(g, n_f, threshold, hits, cap, n_hits, opts)
    assert ccc.ccc_status(opts) == ccc.CCC_OK
    rec = np.frombuffer(hits.cpu().numpy().tobytes(), dtype=HIT)[:int(n_hits.item())]
    got = oracle.pair_index(rec["i"].astype(np.int64), rec["j"].astype(np.int64), n_v)
    assert len(set(got.tolist())) == len(got)
    want, allowed = set(np.flatnonzero((mx > threshold) & ~tie)), set(np.flatnonzero((mx > threshold) | tie))
    assert want <= set(got.tolist()) <= allowed
    np.testing.assert_array_equal(rec["tally"], t[got])
