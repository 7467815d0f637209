"""The default method decides a circuit's route from the gates' patterns: the same route as the blocks'
products give (CPU)."""
import os
import shutil
import subprocess

import pytest

import workloads as W
from conftest import ROOT


@pytest.fixture(scope="module")
def check_exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    exe = tmp_path_factory.mktemp("density") / "block_density_check"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", os.path.join(ROOT, "tests", "block_density_check.cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)
    return exe


FIXED = ["H", "X", "PX", "MX", "PY", "MY", "S"]
CASES = [(14, lambda n: W.random_gate_mix(n, 300, seed=1)), (20, lambda n: W.random_gate_mix(n, 300, seed=2)),
         (16, lambda n: W.random_gate_mix(n, 400, seed=3, two_q_fraction=0.5, names1=FIXED, names2=["CNOT", "CZ"])),
         (13, lambda n: W.random_gate_mix(n, 200, seed=4, two_q_fraction=0.2, names1=FIXED, names2=["CNOT", "SWAP"])),
         (14, W.qft_circuit), (22, W.qft_circuit), (16, lambda n: W.layered_haar_cz(n, 6, 5) + W.qft_circuit(n)),
         (15, lambda n: [("H", (q,), (), None) for q in range(n)] * 2 + W.ghz_circuit(n))]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_patterns_give_the_products_route(check_exe, tmp_path, case):
    import paper_2008_13490_gb300 as qs
    n, make = CASES[case]
    gin = tmp_path / "g.bin"
    qs.gates_array(make(n)).tofile(gin)
    r = subprocess.run([str(check_exe), str(gin), str(n)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
