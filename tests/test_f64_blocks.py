"""complex128 circuits of the default method on the tensor cores (integer slices of FP64).

On the CPU: layout and digit arithmetic of every block; on the GPU: the kernel against the
oracle, and the rows that the integers treat apart (zeros, tiny, not a number)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import ROOT
from oracle import statevector as SV

CIRCUITS = {
    "layered12": (12, lambda n: W.layered_haar_cz(n, 24, 1)),
    "layered13": (13, lambda n: W.layered_haar_cz(n, 20, 2)),
    "layered16": (16, lambda n: W.layered_haar_cz(n, 20, 3)),
    "su4": (15, lambda n: W.layered_su4(n, 6, 4)),
    "scattered": (17, lambda n: [("MAT2", (int(a), int(b)), (), W.haar_su4(W.rng(10 * k + 5)))
                                 for k in range(12) for a, b in W.rng(k).permutation(n)[:16].reshape(-1, 2)]),
}


@pytest.fixture(scope="module")
def check_exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    exe = tmp_path_factory.mktemp("f64") / "f64_block_check"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", os.path.join(ROOT, "tests", "f64_block_check.cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)
    return exe


@pytest.mark.parametrize("name", sorted(CIRCUITS))
def test_layout_and_digits(check_exe, tmp_path, name):
    # inputs and the entry scale round at 2^-54, the result once more: a few 2^-53 of the
    # row's largest amplitude (sums of up to 8 of them in norm); digit sums exact up to 2^24
    import paper_2008_13490_gb300 as qs
    n, make = CIRCUITS[name]
    gin = tmp_path / "g.bin"
    qs.gates_array(make(n)).tofile(gin)
    r = subprocess.run([str(check_exe), str(gin), str(n)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    blocks, worst, big = r.stdout.split()
    assert int(blocks) > 0 and float(worst) <= 8 * 2.0 ** -53 and float(big) <= 2.0 ** 24


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CIRCUITS))
def test_default_method_matches_the_oracle(qs, name):
    # the oracle itself rounds every gate: 2^-53 a gate, independent, on both sides
    n, make = CIRCUITS[name]
    ops = make(n)
    psi0 = W.random_state(n, W.rng(n))
    ref = SV.apply_circuit(psi0.copy(), n, ops)
    st = qs.State(n, qs.QS_C128)
    qs.sv_copy_in(st, psi0)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st)
    st.close()
    assert stats["tile_launches"] == 0 and stats["passes"] > 0
    assert np.linalg.norm(out - ref) <= 2 * np.sqrt(len(ops)) * 2.0 ** -53
    assert np.max(np.abs(out - ref)) <= 1e-12


@pytest.mark.gpu
def test_rows_apart(qs):
    # one dense block on qubits 7..11 of 13: rows are the values of the other bits.  A row of
    # zeros stays exactly zero, rows scaled by 2^-200 give the same digits, a NaN spoils its row
    # only, and a row with one amplitude gives that column of the block
    n = 13
    ops = []
    g = W.rng(7)
    for layer in range(6):
        ops += [("MAT1", (q,), (), W.haar_su2(g)) for q in range(7, 12)]
        ops += [("CZ", (q, q + 1), (), None) for q in range(7 + layer % 2, 11, 2)]
    psi = W.random_state(n, g).reshape(2, 32, 128)   # [bit 12, block columns, row bits 0..6]
    psi[:, :, 3] = 0
    psi[:, :, 4] = psi[:, :, 5] * 2.0 ** -200
    psi[0, 9, 6] = np.nan
    psi[:, :, 8] = 0
    psi[0, 11, 8] = 0.5
    st = qs.State(n, qs.QS_C128)
    qs.sv_copy_in(st, psi.reshape(-1))
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st).reshape(2, 32, 128)
    st.close()
    assert stats["passes"] == 1 and stats["tile_launches"] == 0
    assert np.all(out[:, :, 3] == 0) and np.all(out[1, :, 8] == 0)
    assert np.array_equal(out[:, :, 4], out[:, :, 5] * 2.0 ** -200)
    bad = np.isnan(out.real) | np.isnan(out.imag)
    assert np.all(bad[0, :, 6]) and bad.sum() == 32
    psi[0, 9, 6] = 0
    ref = SV.apply_circuit(psi.reshape(-1).copy(), n, ops).reshape(2, 32, 128)
    ok = ~bad
    assert np.max(np.abs(out[ok] - ref[ok])) <= 1e-15
