"""Which phases are folded into real one-qubit ops: all in a list for one CTA, lone ones in a list for
tile passes (CPU)."""
import os
import shutil
import subprocess

import pytest

import workloads as W
from conftest import ROOT


def _ry_cp(n, layers):
    """RY on every qubit, then CP on alternating neighbour pairs."""
    g = W.rng(1)
    ops = []
    for k in range(layers):
        ops += [("RY", (q,), (g.uniform(-3, 3),), None) for q in range(n)]
        ops += [("CP", (q, q + 1), (g.uniform(-3, 3),), None) for q in range(k % 2, n - 1, 2)]
    return ops


@pytest.fixture(scope="module")
def count(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    import paper_2008_13490_gb300 as qs
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    tmp = tmp_path_factory.mktemp("fold")
    exe = tmp / "fold_rule_dump"
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(ROOT, "tests", "fold_rule_dump.cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)

    def run(ops, n, relabel):
        path = tmp / "gates.bin"
        qs.gates_array(ops).tofile(path)
        r = subprocess.run([str(exe), str(path), str(n), str(int(relabel))], capture_output=True, text=True, check=True)
        return tuple(int(x) for x in r.stdout.split())
    return run


@pytest.mark.parametrize("n,most", [(6, 35), (10, 59), (13, 76)])
def test_lists_for_one_cta_fold_every_phase(count, n, most):
    # a layer's phases go into its neighbours' rotations; the op merge then joins rotations whose
    # choice bits allow it
    assert count(_ry_cp(n, 10), n, False)[0] <= most


def test_fourier_list_for_one_cta(count):
    assert count(W.qft_circuit(10), 10, False)[0] <= 51


@pytest.mark.parametrize("n", [12, 20])
def test_lone_phases_are_folded_in_tile_lists(count, n):
    # at most one rotation per qubit and layer, and no phase of its own but in the last layer
    ops, real, diag = count(_ry_cp(n, 20), n, True)
    assert ops <= 20 * n + n // 2 and diag <= n // 2


@pytest.mark.parametrize("n", [14, 24])
def test_hadamards_beside_runs_of_phases_stay_real(count, n):
    ops, real, diag = count(W.qft_circuit(n), n, True)
    assert real >= n - 2 and diag >= n * (n - 1) // 2 - 4
