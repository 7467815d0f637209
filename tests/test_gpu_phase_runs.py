"""Runs of controlled phases in the tile passes (one register slot, thread jobs, the general
diagonal), the Hadamard gates' gathered factors and the real-matrix ops, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as SV

pytestmark = pytest.mark.gpu


def _circuits(n, g):
    yield "qft", W.qft_circuit(n)
    ops = []   # phases between all places, with every number of Hadamards between them
    for layer in range(3):
        for q in g.permutation(n):
            for _ in range(int(g.integers(0, 4))):
                a, b = (int(x) for x in g.permutation(n)[:2])
                ops.append(("CP", (a, b), (g.uniform(-3, 3),), None))
            ops.append(("H", (int(q),), (), None))
            if g.random() < 0.4:
                ops.append(("CNOT", (int(q), int((q + 1) % n)), (), None))
            if g.random() < 0.3:
                ops.append(("RY", (int(q),), (g.uniform(-3, 3),), None))
    yield "mixed", ops
    # 40 Hadamards on a qubit, a phase between them: the gathered factor is handed on
    yield "deep", [x for k in range(40) for x in (("H", (3,), (), None), ("CP", (3, 5), (0.3,), None))]
    # all qubits against all: more tile x thread phases than register slots
    yield "phases", [("H", (q,), (), None) for q in range(n)] + [
        ("CP", (a, b), (g.uniform(-3, 3),), None) for a in range(n) for b in range(a)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [12, 13, 17])
def test_phase_runs(qs, n, prec):
    g = W.rng(60 + n)
    for name, ops in _circuits(n, g):
        psi = W.random_state(n, W.rng(5))
        st = qs.State(n, prec)
        qs.sv_copy_in(st, psi.astype(st.amp_dtype))
        qs.sv_apply_circuit(st, ops, method=qs.METHOD_TILED)
        out = qs.sv_copy_out(st)
        st.close()
        ref = SV.apply_circuit(psi.copy(), n, ops)
        # every op rounds each amplitude's parts a few times: relative to the norm (1) at most
        # 4 u sqrt(2) per op, u the unit roundoff; and the input's rounding
        u = 2.0 ** -53 if prec else 2.0 ** -24
        assert np.linalg.norm(out - ref) < 6 * u * (len(ops) + 1), name
