"""Log-likelihoods of states with one outcome near certainty: the logarithm keeps its digits however few the counts."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("eps", [1e-12, 1e-10, 1e-6, 1e-3, 0.3, 0.5, 0.6])
@pytest.mark.parametrize("n", [3, 12])
def test_outcomes_near_certainty(qs, n, eps, prec):
    import torch
    st = qs.State(n, prec)
    a = np.zeros(1 << n, dtype=st.amp_dtype)
    a[5], a[2] = math.sqrt(1 - eps), math.sqrt(eps)
    qs.sv_copy_in(st, a)
    p = [float(x.real * x.real) for x in (a[5], a[2])]   # rounded as the state's precision rounds
    for c in [(1, 0), (3, 0), (8, 0), (9, 0), (1000, 0), (0, 2), (7, 1)]:
        counts = np.zeros(1 << n, dtype=np.int32)
        counts[5], counts[2] = c
        got, clamped = qs.sv_loglik(st, torch.from_numpy(counts).cuda())
        ref = math.fsum(k * math.log(q) for k, q in zip(c, p) if k)
        # a logarithm, its product with the count, a sum of two: a few 2^-53 of the result
        assert clamped == 0 and abs(got - ref) <= 8 * 2.0 ** -53 * abs(ref), (c, got, ref)
    st.close()
