"""The packed Box-Muller transform (zo_device.cuh: box_muller_parts, which draws the full-space
pass's normals and Omega of the fp32 panels held in registers) over every uniform of the counter
contract, by the probe and the bound of the plain transform's test; both lanes of a pair, which
have to agree."""
import os
import shutil
import subprocess

import pytest

from parity import NORMAL_ABS

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_packed_box_muller_over_every_uniform(gpu, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "probe")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-DPACKED", "-I", os.path.join(ROOT, "paper_2608_15665_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "harness", "box_muller_probe.cu"), "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    vals = {line.split()[0]: float(line.split()[1]) for line in out.splitlines()}
    print("\n" + out)
    assert vals["bad"] == 0
    bound = 2 * vals["radius"] + max(vals["zcos"], vals["zsin"]) + 2.0 ** -21
    assert bound <= NORMAL_ABS, (bound, out)
