"""The clearance penalty that the rollouts take from double-float arithmetic inside the FP64
band (csrc/terrain.cuh: deck_band), against FP64 (tests/deck_band_check.cpp): whatever it
calls certain has to be FP64's decision and FP64's fp32 value, bit for bit. The heightmap
cell comes from an fp32 position, so positions on node lines, give or take a few fp32
spacings, are where it can be the wrong one; the grid's border, where cells are clamped and
the surface goes on, is among them. It also has to be certain wherever its error bound
allows, or every step along the clearance limit would go to FP64. Runs on the host: g++ and CUDA's headers.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2008_03518_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("g++ or CUDA's headers not found")
    exe = str(tmp_path_factory.mktemp("deck") / "deck_band_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-isystem", include,
                    os.path.join(HERE, "deck_band_check.cpp"), "-o", exe], check=True)
    return exe


N = 1_000_000
GRIDS = [  # nodes per side, box corner, box side, lowest and highest node
    (257, 0.0, 30000.0, 100.0, 200.0),
    (512, 0.0, 30000.0, 0.0, 500.0),
    (64, -5000.0, 10000.0, -50.0, 50.0),
    (1024, 250000.0, 100000.0, 0.0, 2500.0),
    (2, 0.0, 4000.0, 0.0, 300.0),
]


def least_share(nodes, corner, side, low, high):
    """Share of positions that must be certain where the cell is the right one: those above the
    threshold (half of them) unless the clearance is within twice the error bound of it, those
    below also unless the penalty (about 940) is within that of a tie of its fp32 rounding. The
    header's bound, at the far corner."""
    x, H = max(abs(corner), abs(corner + side)) + 7.3, max(abs(low), abs(high))
    slope = 1.0 + 4.0 * H * (nodes - 1) / (0.9 * side)
    z = H + 61.0
    err = 2e-14 * (2 * x + z) * slope + 1e-11 * (H + z + 1000.0) + 1e-12 * slope * 4 * x
    half = 0.5 * 2.0 ** -14
    return 1.0 - 0.5 * min(1.0, 2.0 * err / half) - 4.0 * err / 0.6 - 0.002


@pytest.mark.parametrize("ulps", [0, 1, 8])
@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: f"{g[0]} nodes")
def test_certain_penalties_are_those_of_fp64(checker, grid, ulps):
    r = subprocess.run([checker, str(grid[0] + ulps), str(N), *map(str, grid), str(ulps)], capture_output=True, text=True)
    certain, differ, flips = map(int, r.stdout.split())
    assert (differ, flips, r.returncode) == (0, 0, 0)
    # on lines: each coordinate is on one half of the time, and then in the wrong cell at most half
    assert certain > (1.0 if ulps == 0 else 0.75 ** 2) * least_share(*grid) * N
