"""GPU thresholded 2-way output, SNPs typed on two groups of individuals that hardly overlap (two
chips): a pair's n_ij is then what is left of n_i + n_j - n_f, two large numbers that cancel, and
no pair above the threshold may be dropped however few individuals it shares."""

import numpy as np
import pytest

import oracle
from tests.gpu_util import CCC_RTOL, to_device, workspace

pytestmark = pytest.mark.gpu

HIT = np.dtype([("i", np.int32), ("j", np.int32), ("tally", np.int32, 4), ("ccc", np.float32, 4)])
MISSING = np.uint64(0xAAAAAAAAAAAAAAAA)


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


def _typed(words, lo, hi):
    """The row `words` with every entry outside [lo, hi) missing."""
    out = np.full_like(words, MISSING)
    k = np.arange(len(words), dtype=np.int64) * 32
    a, b = np.clip(lo - k, 0, 32), np.clip(hi - k, 0, 32)
    ones = lambda n: np.array([(1 << (2 * int(x))) - 1 for x in n], dtype=np.uint64)
    keep = ones(b) & ~ones(np.minimum(a, b))
    return (words & keep) | (out & ~keep)


def _panel(n_v, n_f, share, overlap, kind, seed):
    """The first 16 SNPs typed on the first `share` of the individuals, the others on the rest and
    the last `overlap` of those: of the kernel's runs of 16 x 16 pairs most then hold no pair that
    shares more than `overlap`.  Heterozygous wherever typed (every pair then has the value 1/9 at
    gamma 2/3), or codes at random."""
    rng = np.random.default_rng(seed)
    ld = (n_f + 63) // 64 * 2
    cut = int(share * n_f)
    even = np.uint64(0x5555555555555555)
    geno = np.empty((n_v, ld), dtype=np.uint64)
    for i in range(n_v):
        row = np.full(ld, even, dtype=np.uint64)
        if kind == "random":
            lo, hi = rng.integers(0, 1 << 63, (2, ld), dtype=np.int64).astype(np.uint64)
            row = (lo & even) | ((lo & hi & even) << np.uint64(1))  # codes 0, 1, 3
        geno[i] = _typed(row, *((0, cut) if i < 16 else (cut - overlap, n_f)))
    return geno


def _thresholds(mx, n_v, kind):
    """Just below the largest value of one run of 16 x 16 pairs across the two groups."""
    across = [oracle.pair_index(i, j, n_v) for i in range(16) for j in range(16, 32)]
    value = 1.0 / 9.0 if kind == "het" else float(mx[across].max())
    return [float(np.float32(value * (1.0 - below))) for below in (1e-5, 3e-5, 1e-4, 3e-4, 1e-3)]


@pytest.mark.parametrize("kind", ["het", "random"])
@pytest.mark.parametrize("share", [0.4, 0.05])
@pytest.mark.parametrize("n_f,overlap", [(8192, 1), (40000, 2), (200000, 1), (200000, 7), (200000, 64),
                                         (1000000, 2), (1000000, 16), (2097151, 1), (2097151, 33)])
def test_pairs_that_share_few_individuals(n_f, overlap, share, kind):
    import torch

    import paper_1705_08213_gb300 as ccc
    n_v = 41
    geno = _panel(n_v, n_f, share, overlap, kind, seed=n_f + overlap)
    t, c = oracle.ccc2_all(geno, n_f)
    mx = c.max(1)
    g = to_device(geno)
    cap = len(mx)
    hits = torch.zeros(cap * HIT.itemsize, dtype=torch.uint8, device="cuda")
    n_hits = torch.zeros(1, dtype=torch.int64, device="cuda")
    for threshold in _thresholds(mx, n_v, kind):
        tie = np.abs(mx - threshold) <= CCC_RTOL * threshold
        want = set(np.flatnonzero((mx > threshold) & ~tie))
        allowed = set(np.flatnonzero((mx > threshold) | tie))
        assert want
        for operand in (ccc.CCC_OPERAND_E4M3, ccc.CCC_OPERAND_E2M1):
            opts = ccc.ccc_opts_default(operand=operand)
            ws = workspace(ccc.ccc_workspace_size(g, n_f, opts, ccc.CCC_OP_2WAY))
            opts = ccc.ccc_opts_default(operand=operand, workspace=ws)
            ccc.ccc2_filter(g, n_f, threshold, hits, cap, n_hits, opts)
            assert ccc.ccc_status(opts) == ccc.CCC_OK
            rec = np.frombuffer(hits.cpu().numpy().tobytes(), dtype=HIT)[:int(n_hits.item())]
            got = oracle.pair_index(rec["i"].astype(np.int64), rec["j"].astype(np.int64), n_v)
            assert len(set(got.tolist())) == len(got)
            missed = want - set(got.tolist())
            assert not missed, (operand, threshold, len(missed), sorted(missed)[:5])
            assert set(got.tolist()) <= allowed, (operand, threshold)
            np.testing.assert_array_equal(rec["tally"], t[got])
