"""Marginals over masks whose bits lie below, at and above a warp's line of 32 amplitudes, and
log-likelihoods over counts on both sides of the product's limit, against numpy."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,mask", [(1, 0b1), (3, 0b101), (5, 0b10001), (6, 0b100000), (9, 0b101010101), (12, 0b111111111110),
                                    (15, 0b111), (15, 0b111 << 12), (19, 0b1000010000100001000), (20, 0xffff)])
def test_marginals(qs, n, mask, prec):
    # amplitudes that are small integers times 2^-8: probabilities and all their partial sums
    # are exact in either precision, so the marginals are equal, whatever the order
    g = W.rng(100 + n)
    st = qs.State(n, prec)
    a = g.integers(-7, 8, (2, 1 << n))
    qs.sv_copy_in(st, ((a[0] + 1j * a[1]) / 256).astype(st.amp_dtype))
    got, norm = qs.sv_probs(st, fp64=True, marg_mask=mask)
    st.close()
    p = a[0] ** 2 + a[1] ** 2
    K = np.zeros(1 << n, dtype=np.int64)
    for k, b in enumerate(b for b in range(n) if mask >> b & 1):
        K |= (np.arange(1 << n) >> b & 1) << k
    ref = np.zeros(1 << bin(mask).count("1"), dtype=np.int64)
    np.add.at(ref, K, p)
    assert np.array_equal(got.cpu().numpy(), ref / 65536)
    assert norm == p.sum() / 65536


@pytest.mark.parametrize("big,want", [(1.8e19, None), (1e30, np.inf), (np.nan, np.nan)])
def test_marginals_beyond_fp32_sums(qs, big, want):
    # probabilities whose FP32 sum overflows are summed in FP64; infinities and NaN go through
    n = 20   # several lines in one FP32 sum
    st = qs.State(n, 0)
    a = np.zeros(1 << n, dtype=np.complex64)
    a[3::32] = big
    a[4::32] = 0.5
    qs.sv_copy_in(st, a)
    got, norm = qs.sv_probs(st, fp64=True, marg_mask=0b111)
    st.close()
    got = got.cpu().numpy()
    p = np.float64(np.float32(big) * np.float32(big)) * 2 ** 15 if want is None else want
    assert np.array_equal(got, [0, 0, 0, p, 8192, 0, 0, 0], equal_nan=True)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [1, 4, 10, 17])
def test_loglik_counts(qs, n, prec):
    import torch
    g = W.rng(200 + n)
    st = qs.State(n, prec)
    psi = W.random_state(n, g).astype(st.amp_dtype)
    psi[:: 7] *= 1e-18      # probabilities near the smallest normal float, and below it
    psi[3:: 11] = 0
    counts = g.integers(0, 4, 1 << n).astype(np.int32)
    counts[1:: 5] = 8
    counts[2:: 9] = 9
    counts[0] = 100000
    counts[3:: 22] = 0
    qs.sv_copy_in(st, psi)
    got, clamped = qs.sv_loglik(st, torch.tensor(counts, device="cuda"))
    p32 = None if prec else qs.sv_probs(st, fp64=False)[0].cpu().numpy()
    st.close()
    r = psi.view(np.float64 if prec else np.float32)
    # what the kernel sees: the probability in the state's precision (below the smallest normal
    # number its roundings are large against it, so there it has to be the device's own)
    p = r[0::2].astype(np.float64) ** 2 + r[1::2].astype(np.float64) ** 2
    if not prec:
        assert np.all(np.abs(p32 - p) <= p * 2.0 ** -22 + 2.0 ** -148)
        p = p32.astype(np.float64)
    zero = (p <= 0) & (counts > 0)
    ref = np.sum(counts * np.where(counts > 0, np.log(np.where(p > 0, p, 1e-300)), 0))
    assert clamped == zero.sum()
    tol = 1e-12 * abs(ref) if prec else counts.sum() * 2.0 ** -22
    assert abs(got - ref) <= tol, (got, ref)
