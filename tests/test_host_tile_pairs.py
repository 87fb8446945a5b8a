"""How the kernels decode their work items (pairs of query tiles, divisions by multiplication; csrc/s2a_params.h),
checked by host-only C++ programs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2309_12307_b200", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA_INC), reason="needs g++ and the CUDA headers")
@pytest.mark.parametrize("program", ["tile_pairs", "fast_div", "host_plan"])
def test_work_items_decode_to_every_tile_once(tmp_path, program):
    exe = str(tmp_path / program)
    src = os.path.join(ROOT, "tests", "host", program + ".cpp")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", CUDA_INC, src, "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
