"""Launch shape of a z-pass whose tensor map cannot be encoded (here: a spectrum that is not 16-byte aligned): FP32 tiles of 8
columns at 512 rows become 4 columns, with the partial count of that width, because the ordinary kernel would need 768 threads;
every other shape keeps its width and runs without TMA.  Grids and batch slots share the function."""
import os
import shutil
import subprocess
import tempfile

import pytest

pytestmark = pytest.mark.slow

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_03762_gb300", "csrc")
PROGRAM = r"""
#include "gfp_zmap.h"
#include <cstdio>
namespace gfp { bool cz_swizzled(int, int) { return false; } }
int main() {
  alignas(16) static char spec[32];
  for (int n3 : {256, 512})
    for (int mixed = 0; mixed < 2; ++mixed)
      for (int cols : {4, 8}) {
        gfp::Dims d = {};
        d.n1 = 64; d.n2 = 64; d.n3 = n3; d.n1h = 33; d.P = 36; d.N = 64LL * 64 * n3; d.S = 64LL * n3 * d.P;
        gfp::LaunchCfg lc = {};
        lc.x_lines = 1;
        lc.y_cols = 8;
        lc.z_cols = cols;
        lc.z_tma = 1;
        gfp::finalize_cfg(d, lc);
        CUtensorMap m;
        lc.ztmap = &m;
        gfp::attach_ztmap(lc, &m, spec + 1, d, mixed != 0);
        std::printf("%d %d %d %d %d %d\n", n3, mixed, cols, lc.z_cols, lc.z_blocks, lc.ztmap != nullptr);
      }
}
"""


def test_width_without_a_tensor_map():
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as tmp:
        src, exe = os.path.join(tmp, "p.cu"), os.path.join(tmp, "p")
        with open(src, "w") as f:
            f.write(PROGRAM)
        subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, src, "-o", exe],
                       check=True, capture_output=True, text=True)
        out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    for line in out.splitlines():
        n3, mixed, asked, cols, blocks, mapped = map(int, line.split())
        assert mapped == 0
        assert cols == (4 if n3 == 512 and mixed and asked == 8 else asked), line
        assert blocks == -(-33 // cols) * 64, line
    assert len(out.splitlines()) == 8
