"""Marginals of complex64 states in which a large probability meets many small ones: sums as good as FP64's."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mask", [(10, 0b11111), (12, 0b100000000001), (17, 0b1000000000000011)])
@pytest.mark.parametrize("small", [2.0 ** -11.5, 2.0 ** -12.5, 2.0 ** -13.3, 2.0 ** -20, 2.0 ** -30])
def test_small_probabilities_beside_large_ones(qs, n, mask, small):
    # exact sums of the probabilities in the state's precision; FP64 rounds once an addition: 32 in a row
    # and a tree above them
    g = W.rng(n)
    a = (small * (1 + 0.4 * g.random(1 << n))).astype(np.complex64)
    a[::512] = 1
    st = qs.State(n, 0)
    qs.sv_copy_in(st, a)
    p = qs.sv_probs(st, fp64=False)[0].cpu().numpy().astype(np.float64)
    got = qs.sv_probs(st, fp64=True, marg_mask=mask)[0].cpu().numpy()
    st.close()
    bits = [b for b in range(n) if mask >> b & 1]
    K = sum(((np.arange(1 << n) >> b) & 1) << k for k, b in enumerate(bits))
    for k in range(1 << len(bits)):
        ref = math.fsum(p[K == k])
        assert abs(got[k] - ref) <= 48 * 2.0 ** -53 * ref, (k, got[k], ref)
