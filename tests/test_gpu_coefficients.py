"""Coefficients on both sides of the quadrature's boundaries: elements within 24 of the origin (one CTA each),
within 96 (5 points, 13 series terms) and beyond (4 points, 10 terms); gamma = 2 and below.

Tolerance 1e-13 relative, as the coefficient parity elsewhere: each element integral is good to a few FP64
roundings, a_k adds up to eight of them, and a_0 sums all."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N,alpha,gamma", [(2, N, 1.3, 2.0) for N in (2, 24, 25, 26, 96, 97, 98, 130)] +
                         [(2, 120, 0.4, 1.7), (2, 120, 1.9, 2.0), (3, 26, 1.5, 2.0), (3, 30, 0.6, 1.2),
                          (3, 100, 1.0, 2.0)])
def test_coefficients_across_the_rules(frlap, d, N, alpha, gamma):
    from oracle import scheme

    h = 2.0 / N
    a = frlap.frlap_coeffs(d, alpha, gamma, h, (N,) * d).cpu().numpy()
    ref = scheme.coefficients(d, alpha, h, N, gamma)
    assert np.max(np.abs(a - ref) / np.abs(ref)) < 1e-13


def test_diagonal_is_the_rounded_sum(frlap):
    """a_0 = -(sum of all others) - the far field, to one unit in the last place: at h = 2^-10 and alpha = 1.5 the
    scale h^-alpha is a power of two, so the only roundings are the sum's (half a unit) and the far field's."""
    import math

    import numpy as np
    from scipy.integrate import quad

    N, alpha, h = 2048, 1.5, 2.0 ** -10
    a = frlap.frlap_coeffs(2, alpha, 2.0, h, (N, N)).cpu().numpy()
    m = np.where(np.arange(a.shape[0]) > 0, 2.0, 1.0)
    terms = a * m[:, None] * m[None, :]
    terms[0, 0] = 0.0
    far = 4.0 * 2.0 * N ** -alpha / alpha * quad(lambda t: (1 + t * t) ** (-(2 + alpha) / 2), 0.0, 1.0)[0] * 2.0 ** 15
    ref = -math.fsum(terms.ravel().tolist() + [far])
    assert abs(float(a[0, 0]) - ref) <= 2.0 ** -52 * abs(ref)
