"""The wide step and update kernels (twelve threads a site, for lattices with fewer sites than
the GPU has threads) and the runs of steps in one cooperative launch against the kernels with
one thread a site, at ragged volumes (V not a
multiple of the 16, 32 or 64 sites of a block). The two differ in the grouping of the partial
sums only, like two block sizes, so the bar is the one of test_block_sizes: 1e-11."""
import numpy as np
import pytest

import ovinputs as oi
from gpu_util import rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ov():
    import paper_0910_2918_gb300 as ov

    return ov


# (the last one has more two-sided blocks than run at once; there the tuner may take either kernel)
@pytest.mark.parametrize("recomb", [0, 1])
@pytest.mark.parametrize("mu", [0.0, 0.3])
@pytest.mark.parametrize("dims,nrhs,sites", [((5, 4, 7, 6), 1, 16), ((3, 2, 2, 3), 2, 16), ((9, 7, 8, 6), 2, 0)])
def test_wide_equals_narrow(ov, monkeypatch, capfd, dims, nrhs, sites, mu, recomb):
    monkeypatch.setenv("OV_TRACE", "1")
    U = oi.gauge_field(dims, "near_unit", 3, eps=0.35)
    x = np.stack([oi.gaussian_source(dims, 10 + r) for r in range(nrhs)])
    ys = {}
    for bs in (0, 64):
        y = np.zeros_like(x)
        with ov.Overlap(dims, U, -1.5, mu, "df64", opts=ov.make_opts(k_fixed=60, block_size=bs, recombination=recomb)) as op:
            rc, _ = op.sign_apply(x, y, 1e-8, 60, 60)
        assert rc == 0
        ys[bs] = y
    if sites:
        assert f'"wide": {sites}, "one_launch": 1,' in capfd.readouterr().err  # what the tuner took
    for r in range(nrhs):
        assert rel(ys[0][r], ys[64][r]) < 1e-11


def test_wide_batch_equals_narrow(ov):
    shapes = [(4, 4, 4, 4), (5, 3, 4, 6), (6, 6, 4, 4)]
    Us = [oi.gauge_field(d, "near_unit", i, eps=0.3) for i, d in enumerate(shapes)]
    xs = [oi.gaussian_source(d, 20 + i).reshape(1, -1) for i, d in enumerate(shapes)]
    out = {}
    for bs in (0, 64):
        h = ov.ov_batch_create(shapes, Us, [-1.5] * 3, [0.0, 0.2, 0.3], "df64", opts=ov.make_opts(k_fixed=60, block_size=bs))
        out[bs] = [np.zeros_like(x) for x in xs]
        ov.ov_batch_sign_apply(h, xs, out[bs], 1e-8, 60, 60)
        ov.ov_destroy(h)
    for a, b in zip(out[0], out[64]):
        assert rel(a, b) < 1e-11
