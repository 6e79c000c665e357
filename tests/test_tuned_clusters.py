"""The default schedule of the tcgen05 contraction is the same one, with its
clusters dropped where the sectors' tiles would leave them half empty, whether
the autotuner times it or it runs without."""
import os
import shutil
import subprocess

import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_20700_gb300", "csrc")


def test_schedule_of_a_candidate(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path / "tc_candidate_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, "-I", cuda_inc,
                    os.path.join(ROOT, "tests", "cpp", "tc_candidate_check.cpp"),
                    os.path.join(CSRC, "hpsi_tc_plan.cpp"), os.path.join(CSRC, "host_pool.cpp"),
                    "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.gpu
def test_default_schedule_under_the_tuner():
    import paper_2503_20700_gb300 as pkg
    pkg.load()
    n = 10
    h, L = W.cholesky_random(n, 3 * n, seed=4)
    occ, path = W.aufbau_state(h, n, 0)
    default = pkg.tc_shape_candidates()[0]

    def first_product(tune):
        """Energy, schedule and its times after one product of a bond solve."""
        g = pkg.DMRG(h, chol=L, n_elec=n, D=48, precision=pkg.SPLIT_HPSI_TC, max_iter=4, tol=1e-7, occ=occ,
                     two_s_right=path)
        g.sweep(1)
        g.sweep_part(0, n // 2 - 2)
        g.set_tc_autotune(tune)
        r = g.bond_solve(n // 2 - 1, 0, pkg.SPLIT_HPSI_TC, max_iter=1, tol=1e-7, check64=False)
        info = g.tc_schedule()
        g.close()
        return r["energy"], info

    e0, off = first_product(False)
    assert off["shape"] == default and off["cluster"] == 1
    e1, on = first_product(True)
    # the first product of the new histogram was the default's, in the same
    # launch: the same bits
    assert on["ms"][0] > 0 and e1 == e0
