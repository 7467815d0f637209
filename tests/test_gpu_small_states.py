"""Small states (the default method, n < 14): every op kind with its qubits on lanes, warps and CTAs of the
cluster, and op lists around the number staged at a time, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as SV

pytestmark = pytest.mark.gpu


def test_dense_complex64_of_13_qubits(qs):
    ops = W.layered_haar_cz(13, 10, seed=4)
    st = qs.State(13, 0)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st)
    st.close()
    assert stats["passes"] == 1 and stats["tile_launches"] == 0
    ref = SV.apply_circuit(SV.basis(13), 13, ops)
    assert np.linalg.norm(out - ref) < 12 * 2.0 ** -24 * len(ops)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,count", [(1, 20), (2, 60), (4, 300), (5, 100), (6, 100), (7, 300), (8, 300), (9, 900),
                                     (10, 300), (11, 1500), (12, 600), (13, 600)])
def test_small_states(qs, n, count, prec):
    if n == 1:
        ops = [("MAT1", (0,), (), W.haar_su2(W.rng(k))) for k in range(count)]
    else:   # two-qubit ops break the runs of one-qubit ones: about half as many device ops as gates
        ops = W.random_gate_mix(n, count, seed=70 + n, two_q_fraction=0.6)
    psi = W.random_state(n, W.rng(6))
    st = qs.State(n, prec)
    qs.sv_copy_in(st, psi.astype(st.amp_dtype))
    stats = qs.sv_apply_circuit(st, ops)
    if n < 13 or prec:   # (13 complex64 qubits: circuits with dense gates only)
        assert stats["passes"] == 1 and stats["tile_launches"] == 0
    out = qs.sv_copy_out(st)
    st.close()
    ref = SV.apply_circuit(psi.copy(), n, ops)
    # an op rounds each part of an amplitude by at most 4 u of the amplitudes it takes (8 products
    # of two for a dense two-qubit op): relative to the norm (1) 8 sqrt(2) u per op; and the input's
    u = 2.0 ** -53 if prec else 2.0 ** -24
    assert np.linalg.norm(out - ref) < 12 * u * (count + 1)
