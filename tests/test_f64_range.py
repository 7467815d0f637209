"""complex128 blocks of the default method at the edges of their integers' range: matrices and rows that the
integers do not hold give what FP64 arithmetic gives."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import ROOT


def _dense(qubits, layers, g):
    """Haar gates and CZs that make one dense block of five qubits."""
    ops = []
    for layer in range(layers):
        ops += [("MAT1", (q,), (), W.haar_su2(g)) for q in qubits]
        ops += [("CZ", (qubits[i], qubits[i + 1]), (), None) for i in range(layer % 2, 4, 2)]
    return ops


@pytest.fixture(scope="module")
def scale_exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    exe = tmp_path_factory.mktemp("f64s") / "f64_scale_check"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", os.path.join(ROOT, "tests", "f64_scale_check.cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)
    return exe


def test_exponent_fields_of_accepted_blocks(scale_exe):
    # sizes over the range of doubles: a block that is taken keeps every result's exponent field in
    # 1 .. 2046, one that could not is refused
    sizes = [f"{2.0 ** k * f:.17g}" for k in (-900, -120, -101, -90, -61, -60, -59, -1, 0, 40, 58, 59, 60, 90, 99, 900)
             for f in (0.9, 1.0, 1.1)]
    r = subprocess.run([str(scale_exe), *sizes], capture_output=True, text=True, check=True)
    rows = [x.split() for x in r.stdout.splitlines()]
    assert len(rows) == len(sizes)
    taken = [(int(lo), int(hi)) for _, ok, lo, hi in rows if ok == "1"]
    assert taken and all(1 <= lo and hi <= 2046 for lo, hi in taken)
    assert all(ok == "1" for s, ok, _, _ in rows if 2.0 ** -59 <= float(s) <= 2.0 ** 59)


@pytest.mark.gpu
@pytest.mark.parametrize("size,amp", [(9e29, 1e279), (9e29, 1e250), (2e-30, 1e-266), (2e-30, 1.0)])
def test_matrices_far_from_unitary(qs, size, amp):
    # one gate of the block scaled by `size`, amplitudes of about `amp`: results overflow, or leave the
    # normal numbers.  Such circuits run on tile passes, with their values
    n, g = 14, W.rng(11)
    ops = _dense([7, 8, 9, 10, 11], 6, g)
    name, q, par, m = ops[0]
    ops[0] = (name, q, par, m * size)
    psi = W.random_state(n, g) * (amp * 2.0 ** (n / 2))
    outs = []
    for method in (qs.METHOD_AUTO, qs.METHOD_TILED):
        st = qs.State(n, qs.QS_C128)
        qs.sv_copy_in(st, psi)
        stats = qs.sv_apply_circuit(st, ops, method)
        outs.append(qs.sv_copy_out(st))
        st.close()
        assert stats["tile_launches"] > 0
    assert np.array_equal(outs[0].view(np.uint64), outs[1].view(np.uint64)) or \
        np.array_equal(outs[0], outs[1], equal_nan=True)
