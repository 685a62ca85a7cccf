"""GPU thresholded 2-way output of the e4m3 SM-pair tiles, with operand rows and with the codes
expanded in shared memory, each with eight epilogue warps (short vectors) and four (long ones): the
hit list is the oracle's at the edges of tiles, for both normalisations."""

import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import CCC_RTOL, assert_ccc_close, to_device, workspace

pytestmark = pytest.mark.gpu

HIT = np.dtype([("i", np.int32), ("j", np.int32), ("tally", np.int32, 4), ("ccc", np.float32, 4)])


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


@pytest.mark.parametrize("tile", [2, 3])
@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("n_v,n_f,missing", [(2, 70, 0.0), (127, 130, 0.05), (129, 515, 0.4),
                                             (257, 1000, 0.01), (130, 20001, 0.02)])
def test_hits_equal_the_oracle(n_v, n_f, missing, norm, tile):
    import torch

    import paper_1705_08213_gb300 as ccc
    geno = synth.panel_hwe(n_v, n_f, seed=5 * n_v, p_missing=missing, pad_seed=6)
    if n_v > 60:
        synth.plant_near_duplicates(geno, n_f, 20, seed=n_v)
    t, c = oracle.ccc2_all(geno, n_f, norm=norm)
    mx = c.max(1)
    g = to_device(geno)
    cap = len(mx)
    hits = torch.zeros(cap * HIT.itemsize, dtype=torch.uint8, device="cuda")
    n_hits = torch.zeros(1, dtype=torch.int64, device="cuda")
    opts = ccc.ccc_opts_default(norm=norm, tile=tile, operand=ccc.CCC_OPERAND_E4M3)
    ws = workspace(ccc.ccc_workspace_size(g, n_f, opts, ccc.CCC_OP_2WAY))
    opts = ccc.ccc_opts_default(norm=norm, tile=tile, operand=ccc.CCC_OPERAND_E4M3, workspace=ws)
    for threshold in (-1.0, 0.08, 0.155):
        tie = np.abs(mx - threshold) <= CCC_RTOL * abs(threshold)
        ccc.ccc2_filter(g, n_f, threshold, hits, cap, n_hits, opts)
        assert ccc.ccc_status(opts) == ccc.CCC_OK
        rec = np.frombuffer(hits.cpu().numpy().tobytes(), dtype=HIT)[:int(n_hits.item())]
        got = oracle.pair_index(rec["i"].astype(np.int64), rec["j"].astype(np.int64), n_v)
        assert len(set(got.tolist())) == len(got)
        want = set(np.flatnonzero((mx > threshold) & ~tie))
        assert want <= set(got.tolist()) <= set(np.flatnonzero((mx > threshold) | tie))
        np.testing.assert_array_equal(rec["tally"], t[got])
        assert_ccc_close(rec["ccc"], c[got])
