"""The adjoint sweep's runs of one-qubit gates (one op, all derivatives from its four sums), the
diagonals folded into them and the split of passes that hold too many sums, against the oracle's
adjoint; tolerances as for the other gradients of these precisions (test_gpu_grad.py)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import gradient as GR

pytestmark = pytest.mark.gpu


def _runs(n, g):
    """Runs of every make-up on qubits of every place (lane, register, warp, outside the tile)."""
    ang = lambda k: tuple(g.uniform(-3, 3, k))   # noqa: E731
    runs = [
        [("RX", 1), ("RY", 1), ("RZ", 1)],                  # a layer's rotations
        [("RZ", 1), ("U1", 1), ("S", 0)],                   # diagonal alone
        [("U3", 3), ("H", 0), ("U2", 2), ("MAT1", 0)],      # gates without parameters in between
        [("RX", "0")],                                      # U^dagger diagonal, its derivative not
        [("RY", "+"), ("RY", "-")],                         # a product that is the identity
        [("H", 0)],                                         # no derivative
    ]
    ops = []
    for layer in range(3):
        for q in range(n):
            for name, k in runs[(q + layer) % len(runs)]:
                if name == "MAT1":
                    ops.append((name, (q,), (), W.haar_su2(g)))
                elif isinstance(k, str):
                    ops.append((name, (q,), ({"0": 0.0, "+": 0.7, "-": -0.7}[k],), None))
                else:
                    ops.append((name, (q,), ang(k), None))
        for a in range(layer % 2, n - 1, 2):
            kind = ("CZ", "CP", "CNOT", "SWAP")[(a // 2 + layer) % 4] if layer else "CZ"
            ops.append((kind, (a, a + 1) if a % 3 else (a + 1, a), ang(1) if kind == "CP" else (), None))
        ops.append(("CZ", (0, n - 1), (), None))
    return ops


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,ckpt", [(2, 0), (4, 0), (6, 7), (7, 0), (8, 0), (10, 0), (11, 0), (12, 0), (13, 20), (15, 0)])
def test_runs(qs, n, prec, ckpt):
    ops = _runs(n, W.rng(40 + n))
    _check(qs, n, ops, prec, ckpt)


@pytest.mark.parametrize("prec", [0, 1])
def test_more_sums_than_a_pass_holds(qs, prec):
    # one tile, 12 * 9 runs of 4 sums: beyond 352 (complex64) and 196 (complex128) sums
    n, g = 12, W.rng(9)
    ops = []
    for layer in range(9):
        ops += [("RX" if layer % 2 else "RY", (q,), (g.uniform(-3, 3),), None) for q in range(n)]
        ops += [("CNOT", (a, a + 1), (), None) for a in range(layer % 2, n - 1, 2)]
        ops += [("H", (0,), (), None), ("H", (n - 1,), (), None)]
    _check(qs, n, ops, prec, 0)


@pytest.mark.parametrize("prec", [0, 1])
def test_more_sums_than_a_launch_holds(qs, prec):
    # 1200 runs of 4 sums below a tile: beyond 4096
    n, g = 6, W.rng(10)
    ops = []
    for layer in range(200):
        ops += [("RX" if layer % 2 else "RY", (q,), (g.uniform(-3, 3),), None) for q in range(n)]
        ops += [("CNOT", (a, a + 1), (), None) for a in range(layer % 2, n - 1, 2)]
        ops += [("H", (0,), (), None), ("H", (n - 1,), (), None)]
    _check(qs, n, ops, prec, 0)


def _check(qs, n, ops, prec, ckpt):
    w = W.rng(n).normal(size=1 << n)
    Lref, gref = GR.grad_adjoint(ops, n, weights=w)
    st = qs.State(n, prec)
    L, g = qs.sv_grad(st, ops, torch.tensor(w, device="cuda"), mode=0, checkpoint_every=ckpt)
    st.close()
    scale = np.maximum(np.abs(gref), 1.0)
    assert np.max(np.abs(g - gref) / scale) < (1e-9 if prec else 2e-4)
    assert abs(L - Lref) < (1e-10 if prec else 1e-4)
