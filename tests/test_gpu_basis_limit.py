"""Steps beyond the check in hand (speculative ones, and those of the other checks of a group)
that find no basis memory."""
import numpy as np
import pytest

import ovinputs as oi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ov():
    import paper_0910_2918_gb300 as ov

    return ov


@pytest.mark.parametrize("prec,mu,nrhs", [("df64", 0.0, 1), ("df64", 0.3, 1), ("df64", 0.3, 12), ("fp64", 0.3, 2)])
def test_steps_without_basis_memory_leave_the_check_to_decide(ov, monkeypatch, prec, mu, nrhs):
    """The stored basis holds 64 steps. The check at k = 60 ends the run, although the steps run
    beside it would go to 69; a run that does need them gets OV_ERR_NOMEM, and the next apply on
    the handle is bitwise the one without a limit. (The first check has no estimate, so with a
    tolerance of 0.5 the second one ends the run.)"""
    dims = (4, 4, 4, 6)
    U = oi.gauge_field(dims, "near_unit", 0, eps=0.3)
    x = np.stack([oi.gaussian_source(dims, 1 + r) for r in range(nrhs)])
    opts = dict(first_check=50, check_interval=10, recombination=0)
    want = np.zeros_like(x)
    with ov.Overlap(dims, U, -1.6, mu, prec, opts=ov.make_opts(block_size=64, **opts)) as op:
        rc, info = op.sign_apply(x, want, 0.5, 600, 60)
        assert rc == 0 and [i["k"] for i in info] == [60] * nrhs
    monkeypatch.setenv("OV_BASIS_CAP_BYTES", str(64 * 16 * x.size))
    with ov.Overlap(dims, U, -1.6, mu, prec, opts=ov.make_opts(block_size=64, **opts)) as op:
        for tol in (0.5, 1e-10, 0.5, 1e-10, 0.5):
            y = np.zeros_like(x)
            if tol == 0.5:
                rc, info = op.sign_apply(x, y, tol, 600, 60)
                assert rc == 0 and [i["k"] for i in info] == [60] * nrhs
                assert np.array_equal(y, want)
            else:
                with pytest.raises(ov.OvError) as e:
                    op.sign_apply(x, y, tol, 600, 60)
                assert e.value.code == ov.binding.OV_ERR_NOMEM
