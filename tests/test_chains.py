"""Chains of 5-qubit blocks (the default method's sweeps of up to three blocks).

On the CPU the plan and the passes' descriptors, carried out in double precision, reproduce
the circuit; on the GPU the kernel does, against the oracle."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import ROOT
from oracle import statevector as SV

# tiles at the smallest size, runs of every length, blocks on the lowest qubits, scattered
# qubits (single-position boxes), dense two-qubit gates
CIRCUITS = {
    "layered12": (12, lambda n: W.layered_haar_cz(n, 10, 1)),
    "layered13": (13, lambda n: W.layered_haar_cz(n, 12, 2)),
    "layered17": (17, lambda n: W.layered_haar_cz(n, 9, 3)),
    "matching15": (15, lambda n: W.layered_haar_cnot(n, 8, 4)),
    "matching18": (18, lambda n: W.layered_haar_cnot(n, 4, 5)),
    "su4": (16, lambda n: W.layered_su4(n, 5, 6)),
    "mix14": (14, lambda n: W.random_gate_mix(n, 200, 7, two_q_fraction=0.5, names2=["MAT2", "CNOT"])),
    "one_gate": (13, lambda n: [("MAT2", (12, 0), (), W.haar_su4(W.rng(8)))]),
}


@pytest.fixture(scope="module")
def check_exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    exe = tmp_path_factory.mktemp("chains") / "chain_plan_check"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", os.path.join(ROOT, "tests", "chain_plan_check.cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)
    return exe


@pytest.mark.parametrize("name", sorted(CIRCUITS))
def test_plan_and_descriptors_reproduce_the_circuit(check_exe, tmp_path, name):
    import paper_2008_13490_gb300 as qs
    n, make = CIRCUITS[name]
    gin = tmp_path / "g.bin"
    qs.gates_array(make(n)).tofile(gin)
    r = subprocess.run([str(check_exe), str(gin), str(n)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    passes, blocks, err = r.stdout.split()
    assert int(passes) <= int(blocks) <= 3 * int(passes)
    assert float(err) < 1e-11


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CIRCUITS))
def test_default_method_matches_the_oracle(qs, name):
    # relative L2 error: every block rounds each amplitude to FP32 a few times (2^-24 relative
    # each, independent), so sqrt(blocks) * 2^-22 with room for eight such roundings squared
    n, make = CIRCUITS[name]
    ops = make(n)
    psi0 = W.random_state(n, W.rng(n)).astype(np.complex64)
    ref = SV.apply_circuit(psi0.astype(np.complex128), n, ops)
    st = qs.State(n, qs.QS_C64)
    qs.sv_copy_in(st, psi0)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st)
    st.close()
    err = np.linalg.norm(out - ref) / np.linalg.norm(ref)
    assert err <= np.sqrt(max(4, stats["ops_fused"])) * 2.0 ** -22, (err, stats)
    assert abs(np.linalg.norm(out) / np.linalg.norm(psi0) - 1) <= 1e-6
