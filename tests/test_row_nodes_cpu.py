"""The rule behind the row sums of the FP32 kernels: n-node Gauss rules of the
uniform measure on N points sum polynomials of degree 2 n - 1 exactly, and the
node count 2 n = A + 7.2 + 2.6 sqrt(A) + 1.4 D sums a band-limited row."""
import numpy as np
import pytest


def rule(N, n):
    """Golub-Welsch on the discrete Chebyshev recurrence, t_j = (2 j + 1 - N)/N."""
    i = np.arange(1, n)
    b = i * i * (N * N - i * i) / (N * N * (4.0 * i * i - 1.0))
    J = np.diag(np.sqrt(b), 1)
    t, V = np.linalg.eigh(J + J.T)
    return t, N * V[0] ** 2


def points(N):
    return (2 * np.arange(N) + 1.0 - N) / N


@pytest.mark.parametrize("N,n", [(5, 4), (9, 4), (49, 48), (64, 12), (256, 48)])
def test_exact_for_polynomials(N, n):
    t, w = rule(N, n)
    for deg in range(2 * n):
        x = np.polynomial.legendre.Legendre.basis(deg)
        assert abs(np.sum(w * x(t)) - np.sum(x(points(N)))) < 1e-9 * N


@pytest.mark.parametrize("A,D", [(0.0, 0.0), (0.0, 0.6), (0.3, 0.5), (1.0, 0.0), (3.0, 0.1), (10.0, 0.02),
                                 (30.0, 0.01), (65.0, 0.001), (0.1, 11.5)])
def test_node_count_covers_band_limited_rows(A, D):
    """|S|^2 along a row: p0^2 plus parts up to the full swing, of the relative
    sizes the step profile gives them (a few per cent), u exp-like in t."""
    N = 256
    n = int(np.ceil(0.5 * (A + 7.2 + 2.6 * np.sqrt(A) + 1.4 * D)))
    assert n <= 48
    t, w = rule(N, n)

    def f(s):
        u = s if D == 0.0 else np.expm1(D * (s - 1.0)) / D          # |du/dt| <= 1
        return 1.0 + sum(0.03 * np.cos(k / 8 * A * u + k) for k in range(1, 9)) + 0.05 * np.exp(0.2 * u)

    ref = np.sum(f(points(N)))
    assert abs(np.sum(w * f(t)) / ref - 1.0) < 2e-8
