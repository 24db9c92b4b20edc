"""Outer steps in one cooperative launch (small double-float lattices): what the host does when
a wait inside the launch runs out, and where the device refuses the launch; two threads at once."""
import threading
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


# (628 and 384 blocks; a GB300's 152 SMs hold four of the one-sided ones each, two of the two-sided)
@pytest.mark.parametrize("dims,mu,recomb", [((10, 10, 10, 10), 0.0, 0), ((8, 8, 8, 12), 0.3, 0), ((8, 8, 8, 12), 0.3, 1)])
def test_a_refused_launch_becomes_two_launches_a_step(ov, monkeypatch, capfd, dims, mu, recomb):
    """Asked for more blocks than run at once, the device refuses the cooperative launch; the
    steps go on with the wide kernels, here at a size where the tuner takes them, and the answer
    is the one-thread-a-site kernels' to rounding (the bar of the block sizes, 1e-11)."""
    monkeypatch.setenv("OV_TRACE", "1")
    monkeypatch.setenv("OV_ONE_LAUNCH_BLOCKS", "1000000")
    k = 60
    U = oi.gauge_field(dims, "near_unit", 3, eps=0.35)
    x = oi.gaussian_source(dims, 10).reshape(1, -1)
    ys = {}
    for bs in (0, 64):
        ys[bs] = np.zeros_like(x)
        with ov.Overlap(dims, U, -1.5, mu, "df64",
                        opts=ov.make_opts(k_fixed=k, block_size=bs, recombination=recomb)) as op:
            for _ in range(2):
                op.reset_stats()
                assert op.sign_apply(x, ys[bs], 1e-8, k, 60)[0] == 0
            if bs == 0 and '"one_launch": 1' not in capfd.readouterr().err:
                pytest.skip("the tuner took one thread a site")
            assert op.stats()["outer_steps"] == k and op.stats()["graph_launches"] > 0
    assert np.linalg.norm(ys[0] - ys[64]) < 1e-11 * np.linalg.norm(ys[64])


def test_two_handles_in_two_threads(ov):
    """Two threads, each with its own handle and stream, on lattices whose launches do not fit the
    GPU together (256 of 304 blocks each): the same answers, bitwise, as one after the other."""
    import torch

    dims = (8, 8, 8, 8)
    ops, xs, want = [], [], []
    for i in range(2):
        U = oi.gauge_field(dims, "near_unit", i, eps=0.35)
        stream = torch.cuda.Stream()
        ops.append((ov.Overlap(dims, U, -1.5, 0.3, "df64", opts=ov.make_opts(check_interval=10), stream=stream.cuda_stream), stream))
        xs.append(oi.gaussian_source(dims, 5 + i).reshape(1, -1))
        for _ in range(2):  # the first apply tunes
            y = np.zeros_like(xs[i])
            assert ops[i][0].sign_apply(xs[i], y, 1e-9, 800, 100)[0] == 0
        want.append(y)
    bad = []

    def work(i):
        for _ in range(10):
            y = np.zeros_like(xs[i])
            rc, _ = ops[i][0].sign_apply(xs[i], y, 1e-9, 800, 100)
            if rc != 0 or not np.array_equal(y, want[i]):
                bad.append((i, rc))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for op, _ in ops:
        op.close()
    assert not bad
