"""Matrices of a Hadamard gate's shape with large factors, on tile passes: results in the amplitudes' range."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,size,factors", [(0, 1e-34, (1e20, 1e19)), (1, 1e-290, (1e160, 1e149)), (0, 1e-3, (1.0, 0.75, 0.5, 2.0)),
                                               (0, 1e20, (1e-12, 1e-9)), (1, 1.0, (0.7, 0.6, 1e-3))])
def test_factors(qs, prec, size, factors):
    # h [1 1; 1 -1] on neighbouring qubits: each amplitude of the result is a sum of 2^gates of them times the
    # factors, whose product need not be a number of the precision
    n = 14
    had = np.array([[1, 1], [1, -1]], dtype=complex)
    st = qs.State(n, prec)
    psi = (W.random_state(n, W.rng(3)) * 2.0 ** (n / 2) * size).astype(st.amp_dtype)
    ref = psi.astype(np.complex128)
    for q, h in enumerate(factors):
        v = ref.reshape(-1, 2, 1 << q)
        ref = np.stack([v[:, 0] + v[:, 1], v[:, 0] - v[:, 1]], axis=1).reshape(-1) * h
    qs.sv_copy_in(st, psi)
    stats = qs.sv_apply_circuit(st, [("MAT1", (q,), (), had * h) for q, h in enumerate(factors)], qs.METHOD_TILED)
    out = qs.sv_copy_out(st)
    st.close()
    assert stats["tile_launches"] > 0 and np.isfinite(out).all()
    big = np.abs(ref).max()
    u = 2.0 ** -53 if prec else 2.0 ** -24
    # a rounding of the factor, the sum and the product per gate and the input's, of sums of up to 2^gates terms
    assert np.max(np.abs(out / big - ref / big)) <= 4 * u * len(factors) * 2 ** len(factors)
