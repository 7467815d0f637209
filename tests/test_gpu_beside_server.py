"""Small states while a server's persistent kernel holds some SMs or all: the calls do not wait for it to end."""
import time

import numpy as np
import pytest

import workloads as W
from oracle import statevector as SV

pytestmark = pytest.mark.gpu


# (on every SM: states whose kernel needs up to 16 KiB; the shared memory of an SM is divided when the packed
# kernel starts on it)
@pytest.mark.parametrize("n,prec,ctas", [(n, p, 16) for n, p in [(10, 0), (11, 0), (11, 1), (12, 0), (13, 0), (13, 1), (14, 1)]]
                         + [(n, p, 10000) for n, p in [(5, 0), (10, 0), (11, 0), (8, 1), (10, 1)]])
def test_calls_beside_the_packed_kernel(qs, n, prec, ctas):
    # the packed kernel waits up to 40 ms for more work after a circuit; calls made meanwhile take well under
    # half of that (the best of a few: the host is shared)
    ops = W.layered_haar_cz(n, 6, seed=2)
    st = qs.State(n, prec)
    qs.sv_apply_circuit(st, ops)   # buffers
    ref = SV.apply_circuit(SV.basis(n), n, ops)
    srv = qs.Server(persistent_ctas=ctas, idle_ms=40)
    small = W.layered_haar_cz(6, 3, seed=1)
    took = []
    for _ in range(5):
        srv.wait(srv.submit(6, small, 0x3f))
        qs.sv_set_basis(st, 0)
        t0 = time.perf_counter()
        qs.sv_apply_circuit(st, ops)
        out = qs.sv_copy_out(st)
        took.append(time.perf_counter() - t0)
    srv.close()
    st.close()
    assert min(took) < 0.015, took
    u = 2.0 ** -53 if prec else 2.0 ** -24
    assert np.linalg.norm(out - ref) < 12 * u * (len(ops) + 1)


@pytest.mark.parametrize("prec", [0, 1])
def test_gradients_beside_the_packed_kernel(qs, prec):
    n = 9
    ops = [(k, (q,), (0.1 * q + 0.3,), None) for k in ("RX", "RY") for q in range(n)] + [("CZ", (q, q + 1), (), None) for q in range(n - 1)]
    w = W.rng(4).normal(size=1 << n)
    import torch
    weights = torch.tensor(w, device="cuda")
    st = qs.State(n, prec)
    alone = qs.sv_grad(st, ops, weights)
    srv = qs.Server(persistent_ctas=10000, idle_ms=40)
    took = []
    for _ in range(5):
        srv.wait(srv.submit(6, W.layered_haar_cz(6, 3, seed=1), 0x3f))
        t0 = time.perf_counter()
        beside = qs.sv_grad(st, ops, weights)
        took.append(time.perf_counter() - t0)
    srv.close()
    st.close()
    assert min(took) < 0.015, took
    for a, b in zip(alone, beside):
        assert np.allclose(a, b, rtol=0, atol=1e-4 if prec == 0 else 1e-12)
