"""Range of the 2-way popcount path on the host (no GPU): calls of up to 2^31 - 1 tiles of 64 x 64
SNPs are taken, in as many launches as the kernel's 32-SNP tiles need, and every launch's tiles
follow the last one's."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SIDE, GRID = 32, 2 ** 31 - 1


@pytest.fixture(scope="module")
def binary(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc) and shutil.which(nvcc) is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("popc") / "popc_tiles")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1",
                    "-I", os.path.join(ROOT, "paper_1705_08213_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "popc_tiles.cu"), "-o", out], check=True,
                   capture_output=True)
    return out


def coords(t, nB):
    lo, hi = 0, nB - 1  # the last row that starts at or before t
    while lo < hi:
        mid = (lo + hi + 1) // 2
        if mid * nB - mid * (mid - 1) // 2 <= t:
            lo = mid
        else:
            hi = mid - 1
    return lo, lo + t - (lo * nB - lo * (lo - 1) // 2)


@pytest.mark.parametrize("n_v,i0,i1,taken", [
    (2, 0, 2, True), (33, 0, 33, True), (1000, 31, 65, True), (2097120, 0, 2097120, True),
    (2097121, 0, 2097121, True), (2097152, 0, 2097152, True), (3000001, 0, 3000001, True),
    (4194240, 0, 4194240, True), (4194241, 0, 4194241, False), (1 << 26, 0, 1000, True),
    (1 << 26, 5, 64000, True), (1 << 26, 0, 1 << 26, False)])
def test_launches_cover_the_tiles(binary, n_v, i0, i1, taken):
    lines = subprocess.run([binary, str(SIDE), str(n_v), str(i0), str(i1)], check=True,
                           capture_output=True, text=True, timeout=60).stdout.split("\n")
    launches = [tuple(map(int, l.split())) for l in lines if l and not l.startswith("in_range")]
    assert f"in_range {int(taken)}" in lines
    if not taken:
        return
    nB = -(-n_v // SIDE)
    start = lambda r: r * nB - r * (r - 1) // 2
    B0, B1 = i0 // SIDE, -(-i1 // SIDE)
    want = start(B0)
    for k, (first, count, *corners) in enumerate(launches):
        assert first == want and 0 < count <= GRID and (count == GRID or k == len(launches) - 1)
        assert tuple(corners) == coords(first, nB) + coords(first + count - 1, nB)
        want += count
    assert want == start(B1)
