"""Tile passes by the share of their real ops (none, the fewer, half, the most), with and without dense
two-qubit ops and runs of phases, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as SV

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("phases", [False, True])
@pytest.mark.parametrize("real", [0.0, 0.3, 0.5, 0.7, 1.0])
def test_shares_of_real_ops(qs, real, phases, dense, prec):
    n, g = 14, W.rng(31)
    ops = []
    for layer in range(6):
        for q in g.permutation(n):
            q = int(q)
            if g.random() < real:
                name = ["H", "RY", "X"][int(g.integers(0, 3))]
                ops.append((name, (q,), (g.uniform(-3, 3),) if name == "RY" else (), None))
                ops.append(("CNOT", (q, (q + 5) % n), (), None))
            else:
                ops.append(("MAT1", (q,), (), W.haar_su2(g)))
            if phases:
                for r in g.permutation(n)[:3]:
                    if int(r) != q:
                        ops.append(("CP", (q, int(r)), (g.uniform(-3, 3),), None))
        if dense:
            ops.append(("MAT2", (layer, n - 1 - layer), (), W.haar_su4(g)))
    psi = W.random_state(n, g)
    st = qs.State(n, prec)
    qs.sv_copy_in(st, psi.astype(st.amp_dtype))
    stats = qs.sv_apply_circuit(st, ops, method=qs.METHOD_TILED)
    out = qs.sv_copy_out(st)
    st.close()
    assert stats["tile_launches"] > 0
    ref = SV.apply_circuit(psi.copy(), n, ops)
    # an op rounds each part of an amplitude by at most 4 u of the amplitudes it takes (8 products
    # of two for a dense two-qubit op): relative to the norm (1) 8 sqrt(2) u per op; and the input's
    u = 2.0 ** -53 if prec else 2.0 ** -24
    assert np.linalg.norm(out - ref) < 12 * u * (len(ops) + 1)
