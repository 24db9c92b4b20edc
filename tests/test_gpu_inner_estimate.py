"""The inner estimate is held in double: against the two vectors it compares."""
import numpy as np
import pytest

import ovinputs as oi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hermitian", [True, False])
@pytest.mark.parametrize("arith", [0, 1])
def test_inner_estimate_is_held_in_double(hermitian, arith):
    """l = 2 and inner_dl = 1 on 3 x 3 matrices: c' is the c of l = 1, a multiple of e_1, so that the
    inner estimate ||c - c'|| / ||c|| follows from the two c returned with a few roundings. Six on either side of
    2^-53 / sqrt(3) rms each, enlarged by 1 / estimate < 3 where the matrices below are kept,
    leave 12^(1/2) * 3 * 6.4e-17 = 6.7e-16 rms at most, and half of it at the usual estimates of
    ~0.8. Sums in float pairs (2^-48) show above that."""
    import paper_0910_2918_gb300 as ov

    rng = np.random.default_rng(7)
    n = 2048
    A = rng.uniform(0.5, 3.0, (n, 3)) * np.where(rng.random((n, 3)) < 0.5, -1, 1) + 0j
    B = rng.uniform(0.5, 2.0, (n, 3)) + 0j
    G = B.copy()
    if not hermitian:
        A += 0.2j * rng.standard_normal((n, 3))
        G = G * np.exp(0.2j * rng.standard_normal((n, 3)))
    B[:, 0] = G[:, 0] = 0
    U = oi.gauge_field((2, 2, 2, 2), "unit", 0)
    h = ov.ov_create((2, 2, 2, 2), U, -1.5, 0.0, opts=ov.make_opts(inner_dl=1, inner_arith=arith))
    rc, c, est, _ = ov.ov_inner_sign(h, [3] * n, A, B, G, hermitian, 2)
    rc1, c1, _, _ = ov.ov_inner_sign(h, [3] * n, A, B, G, hermitian, 1)
    ov.ov_destroy(h)
    assert rc == 0 and rc1 == 0
    assert np.allclose(abs(c1[:, 0]), 1.0) and np.all(c1[:, 1:] == 0)
    c = c[:, :3].astype(np.clongdouble)
    d = c - c1[:, :3]
    norm = lambda v: np.sqrt((v.real ** 2 + v.imag ** 2).sum(1))
    want = norm(d) / norm(c)
    keep = (want > 1 / 3) & (norm(c) < 3) & np.isfinite(want)
    assert keep.sum() > n // 2
    off = (est[keep] - want[keep]) / want[keep]
    rms = float(np.sqrt(np.mean(off ** 2)))
    assert rms < 3.4e-16
