"""The FP64 sweep's register budget (csrc/cg_kernels.cuh, sweep_min_blocks): in
1D and 2D it asks for three blocks an SM only where the shared memory of three
fits.  Compiled, not run: no GPU needed."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_18042_gb300", "csrc")

SRC = r"""
#include "cg_kernels.cuh"
using namespace cgk;
constexpr int SM = 228 * 1024;
template <int ND, int LW>
constexpr bool three_fit(int more) { return 3 * ((int)sizeof(double) * sweep_smem_doubles<ND, LW>() + more + 2048) <= SM; }
template <int ND, int LW>
constexpr bool sound(int more) { return sweep_min_blocks<ND, true, double, LW>(more) == 2 || three_fit<ND, LW>(more); }
constexpr int TILES = omega_tile_smem<2, double>();  // the persistent stage's sensor tiles
static_assert(sound<1, 4>(0) && sound<1, 8>(0) && sound<2, 4>(0) && sound<2, 8>(0) && sound<2, 16>(0), "sweeps");
static_assert(sound<2, 4>(TILES) && sound<2, 8>(TILES), "persistent stage");
static_assert(sweep_min_blocks<2, true, double, 8>() == 3 && sweep_min_blocks<1, true, double, 8>() == 3, "defaults");
static_assert(sweep_min_blocks<3, true, double, 8>() == 3 && sweep_min_blocks<3, false, double, 4>() == 2, "3D");
static_assert(sweep_min_blocks<2, true, float, 16>() == 4 && sweep_min_blocks<3, true, float, 8>() == 3, "FP32");
"""


def test_blocks_asked_for_fit(tmp_path):
    src = tmp_path / "blocks.cu"
    src.write_text(SRC)
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, "-c", "-o",
                           str(tmp_path / "blocks.o"), str(src)])
