"""A cooperative launch where only a part of the device's SMs can be had (the
launch itself is a stand-in: no GPU)."""
from __future__ import annotations

import subprocess

import pytest

from paper_1602_05232_gb300 import _build

SOURCE = r"""
#include "cc_internal.cuh"
#include <cstdio>
#include <cstdlib>
int main(int, char** argv) {
    const unsigned fits = (unsigned)atoi(argv[1]), grid = (unsigned)atoi(argv[2]);
    unsigned used = 0;
    const cudaError_t e = cc::launch_fitting(grid, [&](unsigned g) {
        if (g > fits) return cudaErrorCooperativeLaunchTooLarge;
        used = g;
        return argv[3][0] == '1' ? cudaErrorInvalidValue : cudaSuccess;
    });
    printf("%d %u\n", (int)e, used);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("fitting")
    (d / "fitting.cu").write_text(SOURCE)
    cmd = [_build._nvcc(), *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", str(_build.INCLUDE),
           "-I", str(_build.CSRC), str(d / "fitting.cu"), "-o", str(d / "fitting")]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("no nvcc")
    assert r.returncode == 0, r.stderr
    return str(d / "fitting")


@pytest.mark.parametrize("fits,grid,broken,want", [
    (608, 608, 0, (0, 608)),       # the whole device
    (607, 608, 0, (0, 304)),
    (64, 608, 0, (0, 38)),
    (1, 608, 0, (0, 1)),
    (1, 1, 0, (0, 1)),
    (0, 608, 0, (720, 0)),         # not one CTA: the error stands
    (64, 608, 1, (1, 38)),         # another error is not retried
])
def test_the_grid_shrinks_until_it_fits(program, fits, grid, broken, want):
    out = subprocess.run([program, str(fits), str(grid), str(broken)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    assert tuple(map(int, out.stdout.split())) == want
