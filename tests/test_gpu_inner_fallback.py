"""The two Roberts-Higham forms of the double-float inner level together: the column by partial
fractions, and the l x l iteration for the matrices that the column leaves (more than 12 steps
needed, or more than rh_maxit); and more matrices than run at a time."""
import numpy as np
import pytest

import ovinputs as oi
from oracle import krylov

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ov():
    import paper_0910_2918_gb300 as ov

    return ov


def tridiagonal(lam, hermitian, rng):
    """(alpha, beta, gamma) of as many (two-sided) Lanczos steps on diag(lam) as it has entries."""
    n = k = len(lam)
    v = rng.uniform(0.5, 1.5, n) + (0 if hermitian else 0.3j * rng.standard_normal(n))
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


def ritz_matrices(count, smallest, hermitian, seed=3, k=8):
    """k x k matrices of an indefinite spectrum in 0.4 .. 4, one eigenvalue of matrix i being smallest(i)."""
    rng = np.random.default_rng(seed)
    out = [np.zeros((count, k), complex) for _ in range(3)]
    for i in range(count):
        lam = np.linspace(0.5, 4.0, k) * rng.uniform(0.9, 1.1, k) * np.where(np.arange(k) % 2, -1.0, 1.0) + 0j
        if not hermitian:
            lam += 0.05j * rng.standard_normal(k)
        lam[0] = smallest(i)
        for dst, src in zip(out, tridiagonal(lam, hermitian, rng)):
            dst[i] = src
    return out


def dense(A, B, G, hermitian):
    H = np.diag(A) + np.diag(B[1:], -1) + np.diag((B if hermitian else G)[1:], 1)
    return H.real if hermitian else H


def handle(ov, **opts):
    return ov.ov_create((2, 2, 2, 2), oi.gauge_field((2, 2, 2, 2), "unit", 0), -1.5, 0.0, opts=ov.make_opts(**opts))


@pytest.mark.parametrize("hermitian", [True, False])
def test_matrices_that_the_column_leaves(ov, hermitian):
    """An eigenvalue of 5e-4 makes one of 2000 of H + H^{-1}: the plain iteration halves it 11 times and
    then converges, more steps than the column takes, so rh_iters > 12 names the l x l iteration;
    with scaling the column does it. Bar: 1e-10, or a hundred times what a relative change of H by
    2^-48, the unit of the float pairs, moves the oracle's vector."""
    count, l = 6, 3
    A, B, G = ritz_matrices(count, lambda i: 5e-4 if i % 2 else 0.5, hermitian)
    refs = []
    for i in range(count):
        H = dense(A[i], B[i], G[i], hermitian)
        N = np.random.default_rng(i).standard_normal(H.shape)
        ref = krylov.nested_sign_e1(H, l, hermitian)[0]
        moved = krylov.nested_sign_e1(H * (1.0 + 2.0 ** -48 * (N + N.T)), l, hermitian)[0]
        refs.append((ref, max(1e-10, 100 * np.linalg.norm(moved - ref))))
        assert refs[-1][1] < 1e-9
    for scaling in (0, 1):
        h = handle(ov, rh_scaling=scaling)
        rc, c, est, its = ov.ov_inner_sign(h, [8] * count, A, B, G, hermitian, l)
        ov.ov_destroy(h)
        assert rc == 0
        for i in range(count):
            assert (its[i] > 12) == (scaling == 0 and i % 2 == 1)
            assert np.linalg.norm(c[i] - refs[i][0]) < refs[i][1]


@pytest.mark.parametrize("hermitian", [True, False])
def test_too_few_steps_allowed_is_an_error(ov, hermitian):
    A, B, G = ritz_matrices(3, lambda i: 0.5, hermitian)
    h = handle(ov, rh_maxit=2)
    rc, _, _, its = ov.ov_inner_sign(h, [8] * 3, A, B, G, hermitian, 3)
    ov.ov_destroy(h)
    assert rc == ov.binding.OV_ERR_RH_NOCONV and list(its) == [2] * 3


@pytest.mark.parametrize("hermitian", [True, False])
def test_more_matrices_than_run_at_a_time(ov, hermitian):
    """1500 problems (3000 matrices with those of the inner estimates, 1216 at a time, some of each
    turn left to the l x l iteration) give bitwise what they give three at a time, and the scratch
    does not grow with them: 600 MB of Roberts-Higham systems, 25 MB of bases and little more."""
    import torch

    count = 1500
    A, B, G = ritz_matrices(count, lambda i: 5e-4 if i % 7 == 0 else 0.5, hermitian)
    free = torch.cuda.mem_get_info()[0]
    h = handle(ov, rh_scaling=0, inner_dl=1)
    rc, c, est, its = ov.ov_inner_sign(h, [8] * count, A, B, G, hermitian, 3)
    used = free - torch.cuda.mem_get_info()[0]
    ov.ov_destroy(h)
    assert rc == 0
    assert used < 700e6
    h = handle(ov, rh_scaling=0, inner_dl=1)
    for i in (0, 3, 602, 606, 609, 1215, 1217, 1497):
        s = slice(i, i + 3)
        rc, c3, est3, its3 = ov.ov_inner_sign(h, [8] * 3, A[s], B[s], G[s], hermitian, 3)
        assert rc == 0
        assert np.array_equal(c3, c[s]) and np.array_equal(est3, est[s]) and list(its3) == list(its[s])
    ov.ov_destroy(h)
