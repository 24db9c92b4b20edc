"""Outer steps in one cooperative launch (small double-float lattices): what the host does when
a wait inside the launch runs out."""
import time

import numpy as np
import pytest

import ovinputs as oi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ov():
    import paper_0910_2918_gb300 as ov

    return ov


@pytest.mark.parametrize("mu", [0.0, 0.3])
@pytest.mark.parametrize("k_fixed", [0, 150])
def test_a_wait_that_runs_out_ends_the_apply(ov, monkeypatch, capfd, mu, k_fixed):
    """With no looks allowed every block but a barrier's last gives up: the apply returns
    OV_ERR_CUDA at its first check, without running on to k_max, and the handle's next apply
    is as before."""
    monkeypatch.setenv("OV_TRACE", "1")
    dims = (6, 4, 4, 4)
    opts = dict(check_interval=5, k_fixed=k_fixed)
    U = oi.gauge_field(dims, "near_unit", 0, eps=0.3)
    x = oi.gaussian_source(dims, 1).reshape(1, -1)
    with ov.Overlap(dims, U, -1.6, mu, "df64", opts=ov.make_opts(**opts)) as op:
        good, after = np.zeros_like(x), np.zeros_like(x)
        assert op.sign_apply(x, good, 1e-9, 600, 100)[0] == 0
        assert '"one_launch": 1' in capfd.readouterr().err
        monkeypatch.setenv("OV_BARRIER_POLLS", "0")
        op.set_opts(**opts)
        for _ in range(2):
            op.reset_stats()
            t0 = time.perf_counter()
            with pytest.raises(ov.OvError) as e:
                op.sign_apply(x, np.zeros_like(x), 1e-9, 600, 100)
            assert e.value.code == ov.binding.OV_ERR_CUDA
            assert time.perf_counter() - t0 < 1.0
            assert op.stats()["checks"] == 1
        monkeypatch.delenv("OV_BARRIER_POLLS")
        op.set_opts(**opts)
        assert op.sign_apply(x, after, 1e-9, 600, 100)[0] == 0
        assert np.array_equal(after, good)
