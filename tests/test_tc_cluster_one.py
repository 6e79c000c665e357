"""CPU check of tcgen05 schedules without clusters, through a small C++ program
(tests/cpp/tc_cluster_one_check.cpp), and (on a GPU) of their products."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_20700_gb300", "csrc")


def test_schedules_without_clusters(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path / "tc_cluster_one_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, "-I", cuda_inc,
                    os.path.join(ROOT, "tests", "cpp", "tc_cluster_one_check.cpp"),
                    os.path.join(CSRC, "hpsi_tc_plan.cpp"), os.path.join(CSRC, "host_pool.cpp"),
                    "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.gpu
@pytest.mark.parametrize("hi", [9, 33, 128, 129])
def test_products_without_clusters(hi):
    """Sectors of one tile each: the default schedule (no clusters) and one in
    clusters (candidate 3, which else only orders the tasks differently)
    against numpy, at the split tolerance of the other tests."""
    import paper_2503_20700_gb300 as pkg
    from test_gpu_dmrg import random_hpsi_problem
    pkg.load()
    rng = np.random.default_rng(hi)
    shapes = [(int(rng.integers(1, hi)), int(rng.integers(1, 2 * hi)),
               [(int(rng.integers(1, hi)), int(rng.integers(1, 3 * hi))) for _ in range(9)]) for _ in range(7)]
    A, P, B, clen, blocks, items, refs = random_hpsi_problem(rng, 0, 0, 0, shapes=shapes)
    C = [np.zeros(clen) for _ in range(2)]
    try:
        for c, cand in zip(C, (0, 3)):
            pkg.set_kernel_tc_shape(cand)
            pkg.ops.hpsi_contract(A, P, B, c, blocks, items, precision=4)
    finally:
        pkg.set_kernel_tc_shape(0)
    for c in C:
        for off, m, n, ref in refs:
            assert np.abs(c[off:off + m * n].reshape(m, n) - ref).max() < 3e-5 * np.abs(ref).max()
