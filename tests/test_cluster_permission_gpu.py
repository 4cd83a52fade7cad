"""Resident launches where the kernel has no permission for clusters of more
than eight blocks, as on a second device (tests/c/cluster_permission.cu)."""
import glob
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_small_lattices_run_without_the_permission_for_large_clusters(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    objects = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    assert objects
    exe = str(tmp_path / "cluster_permission")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                        os.path.join(ROOT, "tests", "c", "cluster_permission.cu"), *objects,
                        "-Xlinker", "--wrap=cudaFuncSetAttribute", "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    run = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout + run.stderr
