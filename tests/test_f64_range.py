"""complex128 blocks of the default method at the edges of their integers' range: matrices and rows that the
integers do not hold give what FP64 arithmetic gives."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import ROOT
from oracle import statevector as SV


def _dense(qubits, layers, g):
    """Haar gates and CZs that make one dense block of five qubits."""
    ops = []
    for layer in range(layers):
        ops += [("MAT1", (q,), (), W.haar_su2(g)) for q in qubits]
        ops += [("CZ", (qubits[i], qubits[i + 1]), (), None) for i in range(layer % 2, 4, 2)]
    return ops


def _compile(tmp_path_factory, name):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from paper_2008_13490_gb300 import _build
    lib = _build.build()
    libdir = os.path.dirname(lib)
    exe = tmp_path_factory.mktemp("f64") / name
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", os.path.join(ROOT, "tests", name + ".cpp"),
                    "-I", os.path.join(ROOT, "paper_2008_13490_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", cuda_inc, "-o", str(exe), "-L", libdir, "-lqsim", f"-Wl,-rpath,{libdir}"],
                   check=True, capture_output=True, text=True)
    return exe


@pytest.fixture(scope="module")
def scale_exe(tmp_path_factory):
    return _compile(tmp_path_factory, "f64_scale_check")


@pytest.fixture(scope="module")
def entry_exe(tmp_path_factory):
    return _compile(tmp_path_factory, "f64_entry_check")


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


def test_entries_of_accepted_blocks_keep_their_digits(entry_exe):
    # five rotations: entries from cos^5 down to sin^5.  An entry of 2^-k of the largest is held to 55 - k
    # bits, and k <= 20 where the block is taken: half a unit of 2^-34 and as much for the reference's scale
    angles = [1e-12, 1e-9, 1e-6, 1e-4, 1e-2, 0.05, 0.1, 0.13, 0.2, 0.5, 1.0, 1.5, 2.0, 3.0, 3.1, 3.1415]
    r = subprocess.run([str(entry_exe), *map(str, angles)], capture_output=True, text=True, check=True)
    rows = [x.split() for x in r.stdout.splitlines()]
    for angle, (_, ok, err) in zip(angles, rows):
        t = min(abs(np.tan(angle / 2)), 1 / abs(np.tan(angle / 2)))   # smallest entry over the largest: t^5
        assert (ok == "1") == (t ** 5 >= 2.0 ** -20), angle
        assert float(err) <= 2.0 ** -34, angle


def _rotations_beside_dense(n, angle):
    """RX by `angle` and CZ on qubits 0..4, Haar gates and CZs on the others."""
    g = W.rng(23)
    small, rest = [], []
    for layer in range(3):
        small += [("RX", (q,), (angle,), None) for q in range(5)]
        small += [("CZ", (q, q + 1), (), None) for q in range(layer % 2, 4, 2)]
    for layer in range(14):
        rest += [("MAT1", (q,), (), W.haar_su2(g)) for q in range(5, n)]
        rest += [("CZ", (q, q + 1), (), None) for q in range(5 + layer % 2, n - 1, 2)]
    return small, rest


@pytest.mark.gpu
@pytest.mark.parametrize("angle", [1e-6, 1e-3])
def test_rare_outcomes_of_small_rotations(qs, angle):
    # The state is a product: for every value of qubits 0..4 that of the others, times an amplitude of about
    # angle^weight.  The rotations' block runs on tile passes (its entries reach down to angle^5), the others
    # as blocks, with every amplitude to its own digits: 2^-34 of a row's amplitudes (kF64Spread) in each of
    # about ten blocks, independent, four times that allowed
    n = 16
    small, rest = _rotations_beside_dense(n, angle)
    st = qs.State(n, qs.QS_C128)
    stats = qs.sv_apply_circuit(st, small + rest)
    out = qs.sv_copy_out(st).reshape(-1, 32)
    st.close()
    assert 0 < stats["tile_launches"] < stats["passes"]
    a = SV.apply_circuit(SV.basis(5), 5, small)
    ref = SV.apply_circuit(SV.basis(n - 5), n - 5, [(k, tuple(q - 5 for q in qq), p, m) for k, qq, p, m in rest])
    for j in range(32):
        assert np.linalg.norm(out[:, j] / a[j] - ref) <= 4 * np.sqrt(10) * 2.0 ** -34, j


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


@pytest.mark.gpu
@pytest.mark.parametrize("qubits", [[9, 10, 11, 12, 13], [0, 1, 2, 3, 4], [1, 4, 6, 9, 13]])
def test_rows_that_the_integers_do_not_hold(qs, qubits):
    # one dense block; rows are the values of the other nine qubits.  Rows of zeros stay zero, a scaled row gives
    # the scaled result, a row with one amplitude gives that column; rows apart (tiny, huge, subnormal, of a
    # wide range, with an infinity or a NaN) give what FP64 gives, and only they
    n, g = 14, W.rng(7)
    ops = _dense(qubits, 6, g)
    others = [q for q in range(n) if q not in qubits]
    J = np.arange(1 << n)
    row = sum(((J >> q) & 1) << k for k, q in enumerate(others))
    col = sum(((J >> q) & 1) << k for k, q in enumerate(qubits))
    at = np.zeros((512, 32), dtype=np.int64)
    at[row, col] = J
    x = W.random_state(n, g)[at] * 2.0 ** (n / 2)
    x[3] = 0
    x[4] = x[5] * 2.0 ** -200
    x[6, 9] = np.nan
    x[7, 20] = np.inf
    x[8] = 0
    x[8, 11] = 0.5
    x[9] = x[5] * 2.0 ** -950          # below the integers' exponents
    x[10] = x[5] * 2.0 ** 1000         # above them
    x[11] = 0
    x[11, 4] = 3e-310                  # subnormal
    x[12:40] = x[5] * np.exp2(-np.arange(32))[g.permutation(32)] ** (np.arange(28)[:, None] / 4)   # ever wider
    x[40, 1:] *= 1e-30
    x[511, 31] = 1e-25
    psi = np.empty(1 << n, dtype=np.complex128)
    psi[at] = x
    st = qs.State(n, qs.QS_C128)
    qs.sv_copy_in(st, psi)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st)[at]
    st.close()
    assert stats["passes"] == stats["ops_fused"] == 1 and stats["tile_launches"] == 0
    assert stats["flops"] == 256.0 * 2 ** n
    # the block, from the oracle's columns
    U = np.stack([SV.apply_circuit(SV.basis(5, j) if j else SV.basis(5), 5,
                                   [(k, tuple(qubits.index(q) for q in qq), p, m) for k, qq, p, m in ops])
                  for j in range(32)], axis=1)
    assert np.all(U != 0)
    assert np.all(out[3] == 0)
    assert np.array_equal(out[4], out[5] * 2.0 ** -200)
    for r in (6, 7):
        assert not np.isfinite(out[r]).any()
    ok = np.array([r for r in range(512) if r not in (6, 7)])
    assert np.isfinite(out[ok]).all()
    # relative to the largest amplitude of the row: 32 products and sums of a few 2^-53 each (the oracle's U
    # as many); subnormal results to their spacing
    want = x[ok] @ U.T
    big = np.abs(x[ok]).max(axis=1, keepdims=True)
    assert np.all(np.abs(out[ok] - want) <= 64 * 2.0 ** -53 * big + 4 * 5e-324 * 32)


@pytest.mark.gpu
def test_small_amplitudes_beside_large_ones(qs):
    # a state whose qubits 0..3 hardly leave zero, then dense blocks on others: each amplitude keeps its own
    # digits (2^-34 of it in each block), also where a block takes idle qubits along
    n, layers, g = 15, 8, W.rng(23)
    t = 1e-4
    small = np.array([1.0 + 0j])
    for q in range(4):
        small = np.kron(np.array([np.cos(t), -1j * np.sin(t)]), small)
    rest = W.random_state(n - 4, g)
    psi = np.kron(rest, small)
    ops = []
    for layer in range(layers):
        ops += [("MAT1", (q,), (), W.haar_su2(g)) for q in range(4, n)]
        ops += [("CZ", (q, q + 1), (), None) for q in range(4 + layer % 2, n - 1, 2)]
    st = qs.State(n, qs.QS_C128)
    qs.sv_copy_in(st, psi)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st).reshape(-1, 16)
    st.close()
    assert stats["passes"] == stats["ops_fused"] and stats["tile_launches"] == 0
    ref = SV.apply_circuit(rest.copy(), n - 4, [(k, tuple(q - 4 for q in qq), p, m) for k, qq, p, m in ops])
    for j in range(16):
        assert np.linalg.norm(out[:, j] / small[j] - ref) <= 4 * np.sqrt(stats["passes"]) * 2.0 ** -34, j
