"""GPU reciprocals and quotients of counts: the reciprocal is the correctly rounded one for every
count and for every sum of tallies up to 2^31, quotients err by at most (1 + 2^-20) 2^-24; and CCC
values of tallies summed over cohorts, past 2^24, stay within the library's error budget."""

import os
import shutil
import subprocess

import numpy as np
import pytest

from tests.gpu_util import assert_ccc_close, workspace

pytestmark = pytest.mark.gpu
# Units of 2^-24 that a value may be off, by (axes, norm): the library's own budget, and past 2^24
# the conversions of the tally (1), of n (1; JOINT 2 more per factor, whose n - gamma R amplifies it
# at most twice) and of each JOINT marginal (2).
BUDGET = {(2, 0): 6, (2, 1): 9, (3, 0): 8, (3, 1): 13}
LARGE = {(2, 0): 2, (2, 1): 10, (3, 0): 2, (3, 1): 14}
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GAMMA = 2.0 / 3.0


@pytest.fixture(scope="module", autouse=True)
def _build():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_08213_gb300 import build
    build.build()


def test_against_cuda_and_exact(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path / "count_quotients")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3",
                    "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1705_08213_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "device", "count_quotients.cu"), "-o", out],
                   check=True, capture_output=True)
    p = subprocess.run([out], check=True, capture_output=True, text=True, timeout=300)
    rcp, rcp_large, quotients, differ, worst = p.stdout.split()
    print(p.stdout)
    assert int(rcp) == 0 and int(rcp_large) == 0
    assert int(quotients) > 100_000_000
    assert float(worst) <= 1.0 + 2.0 ** -20, (worst, differ)


@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("bits", [20, 24, 27, 30])
def test_values_of_summed_tallies(bits, norm):
    """Tables whose sums reach 2^bits and a little more: 2-way and 3-way values in 64 bits."""
    import torch

    import paper_1705_08213_gb300 as ccc
    n_v = 40
    rng = np.random.default_rng(10 * bits + norm)
    alleles = rng.integers(1, 1 << 20, (n_v, 2))
    counts = np.column_stack([2 * alleles[:, 0], 2 * alleles[:, 1], alleles.sum(1)]).astype(np.int32)
    w = 1.0 - GAMMA * counts[:, :2] / (2.0 * counts[:, 2:])
    dev_counts = torch.from_numpy(counts).cuda()
    opts = ccc.ccc_opts_default(norm=norm)
    ws = workspace(ccc.ccc_workspace_size((n_v, 2), 1, opts, ccc.CCC_OP_METRIC))
    opts = ccc.ccc_opts_default(norm=norm, workspace=ws)
    pairs = np.array([(i, j) for i in range(n_v) for j in range(i + 1, n_v)])
    triples = np.array([(i, j, k) for j in range(n_v) for i in range(j) for k in range(j + 1, n_v)])
    for index, axes in ((pairs, 2), (triples, 3)):
        cells = 1 << axes
        t = (rng.random((len(index), cells)) ** 4 * (1 << bits) / cells * 2).astype(np.int64)
        t[0] = 0
        t[1, 1:] = 0
        t[2] = 1 << (bits - axes)
        assert t.sum(1).max() < 1 << 31
        dt = torch.from_numpy(t.astype(np.int32)).cuda()
        dv = torch.full((len(index), cells), -7.0, dtype=torch.float32, device="cuda")
        if axes == 2:
            ccc.ccc2_metric(dt, dev_counts, n_v, opts, dv)
        else:
            ccc.ccc3_metric(dt, dev_counts, n_v, 0, n_v, opts, dv)
        torch.cuda.synchronize()
        cube = t.reshape((len(index),) + (2,) * axes).astype(np.float64)
        over = tuple(range(1, axes + 1))
        n = np.maximum(cube.sum(over, keepdims=True), 1.0)
        want = cube / n
        for x in range(axes):
            shape = [len(index)] + [1] * axes
            shape[x + 1] = 2
            if norm == 1:
                f = 1.0 - GAMMA * cube.sum(tuple(d for d in over if d != x + 1), keepdims=True) / n
            else:
                f = w[index[:, x]].reshape(shape)
            want = want * f
        units = BUDGET[axes, norm] + (LARGE[axes, norm] if bits >= 24 else 0)
        assert_ccc_close(dv.cpu().numpy(), want.reshape(len(index), cells), rtol=units * 2.0 ** -24,
                         what=f"{axes}-way")
