"""The inner level at the edges of its parallel forms: the tridiagonal solves run on 128 lanes
a side with ceil(k / 128) rows each (so k around multiples of 32 and 128, and small k), two-sided
and Hermitian, against the oracle's nested sgn(H) e_1. The bar is that of the inner level's parity
tests, 1e-10, or where the nested vector itself is not that well determined (an inner space of
l = k steps whose basis has lost its orthogonality, a Ritz value close to zero) a hundred times
what a relative change of H by 2^-48, the unit of the float pairs, moves the oracle's vector."""
import numpy as np
import pytest

import ovinputs as oi
from oracle import krylov

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    import paper_0910_2918_gb300 as ov

    h = ov.ov_create((2, 2, 2, 2), oi.gauge_field((2, 2, 2, 2), "unit", 0), -1.5, 0.0)
    yield ov, h
    ov.ov_destroy(h)


def lanczos_coefficients(k, hermitian, seed, n=3000):
    """(alpha, beta, gamma) of k (two-sided) Lanczos steps on a diagonal matrix with an indefinite spectrum."""
    rng = np.random.default_rng(seed)
    lam = rng.uniform(0.4, 5.0, n) * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    lam = lam.astype(complex) if hermitian else lam + 0.05j * rng.standard_normal(n)
    v = rng.standard_normal(n) + (0 if hermitian else 1j) * rng.standard_normal(n)
    v = v.astype(complex) / np.linalg.norm(v)
    w, vp, wp = v.copy(), np.zeros(n, complex), np.zeros(n, complex)
    A, B, G = (np.zeros(k, complex) for _ in range(3))
    for j in range(k):
        p = lam * v - G[j] * vp
        r = lam.conj() * w - np.conj(B[j]) * wp
        A[j] = np.vdot(w, p)
        p, r = p - A[j] * v, r - np.conj(A[j]) * w
        if j + 1 < k:
            d = np.vdot(r, p)
            B[j + 1] = np.sqrt(abs(d))
            G[j + 1] = d / B[j + 1]
            vp, wp, v, w = v, w, p / B[j + 1], r / np.conj(G[j + 1])
    return A, B, G


@pytest.mark.parametrize("hermitian", [True, False])
@pytest.mark.parametrize("ks", [(1, 2, 3, 4), (31, 32, 33, 96), (127, 128, 129, 130), (255, 256, 257, 385), (640, 897, 1000)])
def test_inner_sign_at_chunk_edges(handle, hermitian, ks):
    ov, h = handle
    ld = max(ks)
    A, B, G = (np.zeros((len(ks), ld), complex) for _ in range(3))
    refs = []
    for i, k in enumerate(ks):
        a, b, g = lanczos_coefficients(k, hermitian, 10 * k + hermitian)
        A[i, :k], B[i, :k], G[i, :k] = a, b, g
        H = np.diag(a) + np.diag(b[1:], -1) + np.diag(g[1:], 1)
        H = H.real if hermitian else H
        ref = krylov.nested_sign_e1(H, 120, hermitian)[0]
        rng = np.random.default_rng(k)
        N = rng.standard_normal(H.shape)
        moved = krylov.nested_sign_e1(H * (1.0 + 2.0 ** -48 * (N + N.T)), 120, hermitian)[0]
        refs.append((ref, max(1e-10, 100 * np.linalg.norm(moved - ref))))
    rc, c, est, its = ov.ov_inner_sign(h, list(ks), A, B, G, hermitian, 120)
    assert rc == 0
    for i, k in enumerate(ks):
        ref, bar = refs[i]
        assert np.linalg.norm(c[i, :k] - ref) < bar
        assert np.all(c[i, k:] == 0)
