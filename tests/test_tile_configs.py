"""Register budgets of the tile configurations: CTAs per SM that the launch bounds
promise (compiled, host only). The last two are the 16-point forms that
SRE_ROW13_RB=4 and SRE_STRIDED10_RB=4 build."""
import subprocess

from paper_2601_00761_gb300 import build

SRC = """
#include "sre_internal.cuh"
using namespace sre;
static_assert(TileCfg<float, 13, 0, 5, 1>::MINB == 2, "256 threads x 32 points");
static_assert(TileCfg<float, 12, 0, 6, 1>::MINB == 6, "64 threads x 64 points");
static_assert(TileCfg<float, 10, 0, 5, 1>::MINB == 16, "32 threads x 32 points");
static_assert(TileCfg<float, 14, 0, 5, 1>::MINB == 1, "128 KB");
static_assert(TileCfg<float, 13, 0, 4, 1>::MINB == 2, "512 threads x 16 points, rows");
static_assert(TileCfg<float, 13, 3, 4, 1>::MINB == 2, "512 threads x 16 points, 2^10 rows x 8 columns");
"""


def test_ctas_per_sm(tmp_path):
    src = tmp_path / "cfg.cu"
    src.write_text(SRC)
    cmd = [build.nvcc(), "-std=c++17", "-I", build.CSRC, *build.ARCH, "-c", str(src), "-o", str(tmp_path / "cfg.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
