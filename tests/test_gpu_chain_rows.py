"""What a chain of blocks does with a tile that holds an infinity or a NaN, and sweeps of one, two and three
blocks at the smallest sizes that reach the kernel."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as SV

pytestmark = pytest.mark.gpu


def _block(qubits, layers, g):
    ops = []
    for layer in range(layers):
        ops += [("MAT1", (q,), (), W.haar_su2(g)) for q in qubits]
        ops += [("CZ", (qubits[i], qubits[i + 1]), (), None) for i in range(layer % 2, len(qubits) - 1, 2)]
    return ops


def _run(qs, n, psi, ops):
    st = qs.State(n, qs.QS_C64)
    qs.sv_copy_in(st, psi)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st)
    st.close()
    # the chain kernel and nothing else
    assert stats["tile_launches"] == 0 and stats["launches"] == stats["passes"]
    assert stats["flops"] == 256.0 * 2 ** n * stats["ops_fused"]
    return out, stats


@pytest.mark.parametrize("n", [14, 15])
@pytest.mark.parametrize("blocks", [[[9, 10, 11, 12, 13]], [[0, 1, 2, 3, 4]], [[1, 5, 7, 10, 13]],
                                    [[0, 1, 2, 3, 4], [4, 5, 6, 7, 8]], [[2, 5, 8, 11, 13], [0, 3, 5, 9, 13]],
                                    [[0, 1, 2, 3, 4], [4, 5, 6, 7, 8], [8, 9, 10, 11, 12]],
                                    [[1, 2, 3, 4, 5], [5, 6, 7, 8, 9], [1, 3, 5, 7, 9]]])
def test_short_chains(qs, n, blocks):
    # rounding as in the chains' other tests: a few 2^-24 per block and amplitude
    g = W.rng(n + len(blocks))
    ops = [x for b in blocks for x in _block(b, 6, g)]
    psi = W.random_state(n, g).astype(np.complex64)
    out, stats = _run(qs, n, psi, ops)
    ref = SV.apply_circuit(psi.astype(np.complex128), n, ops)
    assert np.linalg.norm(out - ref) <= np.sqrt(max(4, stats["ops_fused"])) * 2.0 ** -22 * np.linalg.norm(ref)


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e30])
def test_infinities_and_nans_stay_in_their_rows(qs, bad):
    # one block: rows are the values of the other nine qubits, 128 to a tile.  A row that is not finite, or whose
    # squares are not (1e30), leaves the others as accurate as the products are without the norm (FP32
    # accumulation: 2^-20 with room)
    n, qubits = 14, [9, 10, 11, 12, 13]
    g = W.rng(5)
    ops = _block(qubits, 6, g)
    psi = W.random_state(n, g).astype(np.complex64).reshape(32, 512)
    clean = psi.copy()
    psi[7, 100] = bad
    out, _ = _run(qs, n, psi.reshape(-1), ops)
    out = out.reshape(32, 512)
    ref = SV.apply_circuit(clean.reshape(-1).astype(np.complex128), n, ops).reshape(32, 512)
    rest = np.arange(512) != 100
    assert np.isfinite(out[:, rest]).all()
    assert np.linalg.norm((out - ref)[:, rest]) <= 2.0 ** -20
    if not np.isfinite(bad):
        assert not np.isfinite(out[:, 100]).any()
