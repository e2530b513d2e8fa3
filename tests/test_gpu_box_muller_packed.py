"""The packed Box-Muller transform (zo_device.cuh: box_muller_parts, the full-space pass's and
the fp32 bases' draws) over every uniform of the counter contract, by the probe and the bound of
the plain transform's test; both lanes of a pair, which have to agree."""
import os
import shutil
import subprocess

import pytest

from parity import NORMAL_ABS

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PACKED = """#include "zo_device.cuh"

// the transform of one pair of words in both lanes; a NaN where they differ
__device__ float2 packed(uint32_t xa, uint32_t xb) {
  const uint32_t a[2] = {xa, xa}, b[2] = {xb, xb};
  float2 nr[1], c[1], s[1];
  zo::box_muller_parts<1, float2>(a, b, nr, c, s);
  const float2 z0 = zo::mul2(nr[0], c[0]), z1 = zo::mul2(nr[0], s[0]);
  return z0.x == z0.y && z1.x == z1.y ? make_float2(z0.x, z1.x) : make_float2(nanf(""), nanf(""));
}
"""


def test_packed_box_muller_over_every_uniform(gpu, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    with open(os.path.join(ROOT, "tests", "harness", "box_muller_probe.cu"), encoding="utf-8") as f:
        text = f.read()
    assert text.count('#include "zo_device.cuh"\n') == 1 and text.count("zo::box_muller(") == 2
    text = text.replace('#include "zo_device.cuh"\n', PACKED).replace("zo::box_muller(", "packed(")
    # a NaN is no error in "d > max": make it one
    text = text.replace("if (dr > e_rad)", "if (!(dr <= e_rad))").replace(
        "if (dc > e_c)", "if (!(dc <= e_c))").replace("if (ds > e_s)", "if (!(ds <= e_s))")
    src, exe = tmp_path / "probe.cu", str(tmp_path / "probe")
    src.write_text(text, encoding="utf-8")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-I", os.path.join(ROOT, "paper_2608_15665_gb300", "csrc"), str(src), "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    vals = {line.split()[0]: float(line.split()[1]) for line in out.splitlines()}
    print("\n" + out)
    bound = 2 * vals["radius"] + max(vals["zcos"], vals["zsin"]) + 2.0 ** -21
    assert bound <= NORMAL_ABS, (bound, out)
