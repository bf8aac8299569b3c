"""The learned start's dense layers on the tensor cores (exact bfloat16 pieces of the float32 rows)
at row counts around their 16-row and 64-row tiles, from one row to several tiles per block.

Three layers of at most 130 + 30 float32 roundings (6e-8 each) and their backward: 3e-5 in the
2-norm at worst, against the float64 oracle."""
import numpy as np
import pytest

import lpgen
from oracle import gnn_oracle as G
from test_gpu_gnn import P, biased_params, labels  # noqa: F401  (P: the fixture)

pytestmark = pytest.mark.gpu

TOL = 3e-5


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("m,n", [(1, 2), (15, 17), (16, 32), (31, 33), (63, 65), (64, 128),
                                 (129, 191), (3000, 20011)])
def test_dense_layers_at_tile_edges(P, m, n):  # noqa: F811
    lp = lpgen.random_sparse_lp(m + n, m, n, density=min(1.0, 6.0 / m))
    theta = biased_params(m)
    md = P.GnnModel(seed=0)
    md.set_params(theta)
    xs, ys = labels(lp, n)
    g = md.graph(lp, xs, ys)
    x, y, _ = md.forward(g)
    xr, yr = G.predict(theta.astype(np.float64), lp)
    assert rel(x, xr) <= TOL and rel(y, yr) <= TOL, (rel(x, xr), rel(y, yr))
    md.zero_grad()
    md.backward(g, scale=1.0)
    ycanon = np.where(lp.sense == ord("L"), -ys, ys)
    _, want = G.grad(theta.astype(np.float64), G.graph(lp), xs, ycanon)
    assert rel(md.grad(), want) <= TOL, rel(md.grad(), want)


def test_gradient_sums_beyond_the_range_of_float32(P):  # noqa: F811
    """Labels of 3e36 in the first half of the rows and -3e36 in the second: the partial sums of a
    head weight's gradient leave the range of float32 on the way to a sum within it.  (TOL of the sum
    of the terms' magnitudes.)"""
    n = 4096
    lp = lpgen.random_sparse_lp(3, 64, n, density=0.02)
    lp.l[:], lp.u[:] = 0.0, np.inf
    theta = biased_params(5)
    d = G.unpack(theta.astype(np.float64))
    for name, _ in G.param_shapes():
        if name.startswith("b"):
            d[name] *= 8.0
    theta = G.pack(d).astype(np.float32)
    xs, ys = labels(lp, 1)
    xs = np.where(np.arange(n) < n // 2, 3e36, -3e36)
    md = P.GnnModel(seed=0)
    md.set_params(theta)
    g = md.graph(lp, xs, ys)
    md.zero_grad()
    md.backward(g, scale=1.0)
    graph = G.graph(lp)
    h = G.forward(theta.astype(np.float64), graph, keep=True)[2]["hv"][-1]
    ycanon = np.where(lp.sense == ord("L"), -ys, ys)
    _, want = G.grad(theta.astype(np.float64), graph, xs, ycanon)
    got = G.unpack(md.grad().astype(np.float64))["w_x"]
    want = G.unpack(want)["w_x"]
    terms = 3e36 * 2.0 / n * h.sum(axis=0)
    top = float(np.finfo(np.float32).max)
    assert np.max(0.5 * terms) > 1.1 * top and np.max(np.abs(want)) < 0.9 * top
    assert np.all(np.isfinite(got))
    assert np.all(np.abs(got - want) <= TOL * terms)


def test_weight_gradients_are_not_cut_towards_zero(P):  # noqa: F811
    """Both operands of a weight gradient are truncated into pieces, so a product of small pieces that
    is left out has the sign of its term: with terms of one sign (labels far below the predictions)
    the smallest three products are 2^-24 of the sum on average.  Exact products leave no such bias:
    under a quarter of that, over the layers' weights of four graphs."""
    cut = []
    for seed in range(1, 5):
        lp = lpgen.set_cover(seed, m=3000, n=12000)
        rng = np.random.default_rng(seed)
        xs, ys = rng.random(lp.n) - 5.0, rng.random(lp.m) + 5.0 * float(np.max(np.abs(lp.c)))
        theta = biased_params(seed)
        md = P.GnnModel(seed=0)
        md.set_params(theta)
        g = md.graph(lp, xs, ys)
        md.zero_grad()
        md.backward(g, scale=1.0)
        _, want = G.grad(theta.astype(np.float64), G.graph(lp), xs, ys)
        got, want = G.unpack(md.grad().astype(np.float64)), G.unpack(want)
        for k in want:
            if k.startswith("W_") and k[-1].isdigit():
                cut.append(np.sum((got[k] - want[k]) * np.sign(want[k])) / np.sum(np.abs(want[k])))
    assert np.mean(cut) > -0.25 * 2.0 ** -24, np.mean(cut)
