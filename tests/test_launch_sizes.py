"""Blocks per system of the batched Krylov passes (host rule)."""
import shutil
import subprocess

import pytest

from paper_1705_08849_gb300 import build

MAIN = r"""
#include <cstdio>
#include "fit_residency.cuh"
int main() {
  int per_sm, nsm, batch, least;
  long long most;
  while (std::scanf("%d %d %d %d %lld", &per_sm, &nsm, &batch, &least, &most) == 5)
    std::printf("%lld\n", fit_blocks_per_system(per_sm, nsm, batch, least, most));
}
"""


def test_blocks_per_system(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    (tmp_path / "main.cpp").write_text(MAIN)
    cuda = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-I", build.CSRC, "-I", cuda.rsplit("/", 2)[0] + "/include",
                    str(tmp_path / "main.cpp"), "-o", str(tmp_path / "main"), "-Wl,--unresolved-symbols=ignore-all"],
                   check=True)
    rows = [(p, 152, b, least, most) for p in (2, 4, 8) for b in (1, 2, 3, 8, 16, 17, 64, 1000, 4096) for least in (38, 152)
            for most in (0, 1, 7, 38, 151, 152, 1216)]
    r = subprocess.run([str(tmp_path / "main")], input="\n".join(" ".join(map(str, q)) for q in rows), text=True,
                       capture_output=True, check=True)
    for (p, nsm, b, least, most), n in zip(rows, map(int, r.stdout.split()), strict=True):
        assert 1 <= n <= max(1, most)  # never more than the buffers hold
        # every system has its least share, however many share the call; one system has all that is resident
        assert n >= min(most, least) and n >= min(most, p * nsm // b)
        if b == 1:
            assert n == max(1, min(most, max(least, p * nsm)))
