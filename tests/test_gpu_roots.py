"""FP64 square root and the two-step reciprocal forms against the IEEE operations, on the device."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.gpu
def test_roots_and_two_step_forms(tmp_path):
    """sqrt_nr: the correction leaves a quarter of an ulp of the product x y and its own half, so
    within an ulp, and the IEEE root outside the seed's range; the reciprocal within an ulp, its
    root within two of 1/sqrt(x) (itself two roundings), the quotient IEEE."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "root_check")
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2508_16387_gb300", "csrc"),
                    os.path.join(HERE, "native", "root_check.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    got = {line.rsplit(" ", 1)[0]: float(line.rsplit(" ", 1)[1]) for line in r.stdout.splitlines()}
    assert got["sqrt worst ulp"] <= 1.0 and got["rcp worst ulp"] <= 1.0 and got["rsqrt worst ulp"] <= 2.0, got
    assert got["special roots differing"] == 0 and got["quotients differing"] == 0, got
