"""Host-side check of the sweep kernel's work lists, no GPU: nvcc builds
tests/sweep_plan_check.cu (which includes the library's ibs_sweep.cu) and runs
it on the CPU: 16 sample counts x 10 marker counts x 4 cluster counts, 60 batches
x 2, 400 serving steps and as many unbatched requests; and the lengths and the
kinds of serving steps."""
import os
import subprocess

import pytest

from test_work_lists import ROOT, _nvcc


def test_sweep_plans_cover_the_triangle(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "sweep_plan_check")
    build = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                            "-I", os.path.join(ROOT, "include"), "-o", exe,
                            os.path.join(ROOT, "tests", "sweep_plan_check.cu")],
                           capture_output=True, text=True, timeout=600)
    assert build.returncode == 0, build.stdout + build.stderr
    run = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout[-4000:]
    assert "checked 1560 lists, 0 failures" in run.stdout, run.stdout[-2000:]
