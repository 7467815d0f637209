"""Calls whose kernels want large scratch buffers, on an allocator that refuses them: the ways that need less."""
import numpy as np
import pytest

import workloads as W
from oracle import statevector as SV

pytestmark = pytest.mark.gpu


@pytest.fixture
def limited(qs, monkeypatch):
    """A state whose allocator hands out no more than `limit` bytes at a time once it is made."""
    full = qs.torch_allocator()
    limit, refused = [None], []

    @qs._ALLOC_T
    def alloc(nbytes, stream, ctx):
        if limit[0] is not None and nbytes > limit[0]:
            refused.append(nbytes)
            return None
        return full.alloc(nbytes, stream, ctx)

    a = qs._Allocator(alloc, full.free, None)
    a._keep = (alloc, full)
    monkeypatch.setattr(qs, "torch_allocator", lambda: a)

    def make(n, prec, most):
        limit[0] = None
        st = qs.State(n, prec)
        limit[0] = most
        refused.clear()
        return st, refused
    yield make
    limit[0] = None


@pytest.mark.parametrize("n,count", [(14, 0), (16, 0), (12, 1500), (13, 1500)])
def test_circuits(qs, limited, n, count):
    # 16 qubits: dense blocks with 64 KiB each; 12 and 13: the op list of the registers' kernel.  Tile passes
    # carry ops other than phases with the launch
    ops = W.random_gate_mix(n, count, seed=n, two_q_fraction=0.6, names1=["MAT1"], names2=["MAT2"]) if count else W.layered_haar_cz(n, 12, seed=n)
    st, refused = limited(n, qs.QS_C128, 192 << 10)
    stats = qs.sv_apply_circuit(st, ops)
    out = qs.sv_copy_out(st)
    st.close()
    assert refused and stats["tile_launches"] > 0
    assert np.linalg.norm(out - SV.apply_circuit(SV.basis(n), n, ops)) < 12 * 2.0 ** -53 * (len(ops) + 1)


@pytest.mark.parametrize("prec", [0, 1])
def test_gradients(qs, limited, prec):
    import torch
    n = 10
    ops = [(k, (q,), (0.1 * q + 0.3,), None) for k in ("RX", "RY", "RZ") for q in range(n)] + \
        [("CZ", (q, q + 1), (), None) for q in range(n - 1)]
    w = torch.tensor(W.rng(4).normal(size=1 << n), device="cuda")
    st = qs.State(n, prec)
    ref = qs.sv_grad(st, ops, w)
    st.close()
    st, refused = limited(n, prec, 64 << 10)
    got = qs.sv_grad(st, ops, w)
    st.close()
    assert refused
    for a, b in zip(ref, got):
        assert np.allclose(a, b, rtol=0, atol=1e-4 if prec == 0 else 1e-12)
