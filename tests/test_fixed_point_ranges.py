"""Ranges of the FP64 passes' 64-bit fixed-point transforms, for every radix schedule the library accepts: no element leaves 63
bits, and a line is scaled down by no more than it can grow.

A line enters with |re|, |im| <= 2^60, a modulus of 2^60.5.  A radix-R layer multiplies the modulus by at most R; the elements
shrink between the layers of the composite radices (fx_inner) and between stages (post).  The twiddle product's middle sums are at
most 2^31.5 |a| / 2^32 + 2^31.5 2^30 for an element a, below 2^63 for |a| <= 2^62.85.

Scaled down by S bits in all, a line of length n ends in units of 2^(S - 60) of its largest element, whatever it grows to:
with S beyond log2 n even a line that grows by n would lose bits.  0.3 leaves room for whole bits."""
import math
import os
import shutil
import subprocess
import tempfile

import pytest

pytestmark = pytest.mark.slow

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_03762_gb300", "csrc")
LAYERS = {2: (2,), 3: (3,), 4: (4,), 6: (3, 2), 8: (4, 2), 9: (3, 3), 12: (4, 3), 16: (4, 4), 18: (3, 3, 2)}
PROGRAM = r"""
#include "gfp_fx.cuh"
#include <cstdio>
int main() {
  gfp::FftPlan p;
  while (std::scanf("%d", &p.nst) == 1) {
    p.n = 1;
    for (int s = 0; s < p.nst; ++s) { if (std::scanf("%d", &p.radix[s]) != 1) return 1; p.n *= p.radix[s]; }
    const gfp::FftPlan m = gfp::fx_plan(p);
    std::printf("%d %d", p.n, gfp::fx_shift(m));
    for (int s = 0; s < m.nst; ++s) std::printf(" %d %d %d", m.radix[s], gfp::fx_inner(m.radix[s]), (int)(m.post >> (2 * s) & 3));
    std::printf("\n");
  }
}
"""


def _schedules(done=(), prod=1):
    if done:
        yield done
    for r in (2, 3, 4, 8, 16):
        if prod * r <= 1024 and len(done) < 12:
            yield from _schedules(done + (r,), prod * r)


def test_every_schedule_stays_in_range_and_keeps_its_bits():
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as tmp:
        src, exe = os.path.join(tmp, "p.cu"), os.path.join(tmp, "p")
        with open(src, "w") as f:
            f.write(PROGRAM)
        subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-Xcicc", "-O0", "-Xptxas", "-O0",
                        "-I", CSRC, src, "-o", exe], check=True, capture_output=True, text=True)
        text = "\n".join("%d %s" % (len(s), " ".join(map(str, s))) for s in _schedules())
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout
    lines = set(out.splitlines())
    assert len(lines) > 100
    for line in lines:
        n, shift, *rest = map(int, line.split())
        stages = [rest[i:i + 3] for i in range(0, len(rest), 3)]
        bits, total = 60.5, 0
        for i, (radix, inner, _) in enumerate(stages):
            scales = ([stages[i - 1][2]] if i else [0])  # before the stage, then between its layers
            layers = LAYERS[radix]
            scales += {1: [], 2: [inner], 3: [2, inner - 2]}[len(layers)]
            for down, grow in zip(scales, layers):
                assert bits <= 62.85, line  # into the twiddle product or the shift
                bits += math.log2(grow) - down
                total += down
                assert bits < 63.0, line
        assert total == shift, line
        assert shift <= math.log2(n) + 0.3, line
