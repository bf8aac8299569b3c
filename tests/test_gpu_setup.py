"""The device setup at the row lengths and sizes where its kernels change their path.

The scaling passes walk rows longer than 256 entries (and 8 average rows) by whole blocks, a
sum in rounds of 896 terms; shorter rows in tiles of up to 256 rows.  The factors feed the
float64 iteration, so ten fixed steps against the oracle show an error in any of them: the
oracle's factors and steps round differently by a few units in the last place of values of
order one, 1e-12 leaves four digits over that.
"""
import numpy as np
import pytest

import lpgen
from oracle import pdlp_oracle as O

pytestmark = pytest.mark.gpu

FIXED = dict(iter_limit=10, adaptive_step=0, restarts=0, terminate=0, fixed_eta=0.9)


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as G
    G.build()
    import paper_2503_10344_gb300 as P
    return P


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(1.0, np.linalg.norm(b)))


def long_lp(length, m, n, ones, seed):
    """Rows and columns of one to three entries, then one row and one column of `length`."""
    rng = np.random.default_rng(seed)
    rows, cols = [np.arange(m)], [rng.integers(0, n, m)]
    rows.append(rng.integers(0, m, n))
    cols.append(np.arange(n))
    keep = (rows[1] != m // 2)
    rows[1], cols[1] = rows[1][keep], cols[1][keep]
    rows.append(np.full(length, m // 2))
    cols.append(rng.choice(n, length, replace=False))
    if length <= m:
        rows.append(rng.choice(m, length, replace=False))
        cols.append(np.full(length, n // 3))
    key = np.unique(np.concatenate(rows) * n + np.concatenate(cols))
    rows, cols = key // n, key % n
    val = np.ones(key.size) if ones else rng.uniform(0.1, 3.0, key.size) * rng.choice([-1, 1], key.size)
    ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    return lpgen.LP(m, n, ptr.astype(np.int64), cols.astype(np.int32), val, rng.uniform(0.5, 1, m),
                    np.full(m, lpgen.SENSE_GE, dtype=np.uint8) if ones else
                    rng.choice([lpgen.SENSE_GE, lpgen.SENSE_LE, lpgen.SENSE_EQ], m).astype(np.uint8),
                    rng.uniform(-1, 1, n), np.zeros(n), np.ones(n), np.zeros(n, dtype=np.uint8))


@pytest.mark.parametrize("length,m,n", [(256, 700, 900), (257, 257, 513), (896, 897, 3000),
                                        (897, 2000, 1000), (4097, 300, 6000), (17520, 20000, 19000)])
@pytest.mark.parametrize("prec,ones", [("fp64", False), ("fp64", True), ("bf16", True)])
def test_scaling_of_long_rows_and_columns(P, length, m, n, prec, ones):
    lp = long_lp(length, m, n, ones, length)
    _, _, r, it = P.pdlp_solve(lp, P.default_params(precision=prec, **FIXED), iterates=True)
    ref = O.solve(lp, O.Params(iter_limit=10, adaptive=False, restarts=False, terminate=False,
                               fixed_eta=0.9))
    # float32 iterates: ten steps of a few float32 roundings each
    tol = 1e-12 if prec == "fp64" else 5e-6
    for k in ("x_cur", "y_cur", "x_avg", "y_avg"):
        assert rel(it[k], getattr(ref, k)) <= tol, (k, rel(it[k], getattr(ref, k)))
    assert r["omega"] == pytest.approx(ref.omega, rel=1e-12)


@pytest.mark.parametrize("count", [1, 3])
def test_batch_scalars_and_scaling(P, count):
    """The scalars and factors of each LP of a batch against the oracle's, one LP at a time."""
    lps = [long_lp(300 + 600 * k, 800 + k, 2000 - k, False, k) for k in range(count)]
    xs, ys, res = P.pdlp_solve_batch(lps, P.default_params(**FIXED))
    for lp, x, y, r in zip(lps, xs, ys, res):
        ref = O.solve(lp, O.Params(iter_limit=10, adaptive=False, restarts=False, terminate=False,
                                   fixed_eta=0.9))
        assert r["omega"] == pytest.approx(ref.omega, rel=1e-12)
        assert rel(x, ref.x) <= 1e-12 and rel(y, ref.y) <= 1e-12


@pytest.mark.parametrize("m,n", [(2047, 2048), (2048, 2049), (2049, 4096), (4097, 10_240)])
def test_prefix_sums_at_tile_edges(P, m, n):
    """Row and column counts around the 2,048 counts of a scan's tile: one launch, two, the last
    tile full or of one count.  Twenty float64 steps agree with the oracle's to rounding."""
    lp = lpgen.random_sparse_lp(m, m, n, density=3.0 / m)
    kw = dict(iter_limit=20, adaptive_step=0, restarts=0, terminate=0, fixed_eta=0.5)
    _, _, _, it = P.pdlp_solve(lp, P.default_params(**kw), iterates=True)
    ref = O.solve(lp, O.Params(iter_limit=20, adaptive=False, restarts=False, terminate=False, fixed_eta=0.5))
    for k in ("x_cur", "y_cur"):
        want = getattr(ref, k)
        assert np.linalg.norm(it[k] - want) <= 1e-12 * max(1.0, np.linalg.norm(want)), k


@pytest.mark.parametrize("lanes", [2, 4])
def test_long_row_cutoff(P, lanes):
    """Rows and columns on both sides of 64 entries per lane, the cut-off to a block per row."""
    rng = np.random.default_rng(lanes)
    cut, n = 64 * lanes, 900
    lengths = np.array([cut - 1, cut, cut + 1, 1, 3] * 12)
    m = len(lengths)
    rows = np.repeat(np.arange(m), lengths)
    cols = np.concatenate([rng.choice(n, k, replace=False) for k in lengths])
    lp = lpgen._lp(m, n, rows, cols, rng.integers(1, 4, rows.size).astype(float), rng.uniform(0, 2, m),
                   rng.choice([lpgen.SENSE_GE, lpgen.SENSE_LE, lpgen.SENSE_EQ], m),
                   rng.uniform(-1, 1, n), np.zeros(n), rng.uniform(1, 5, n), np.zeros(n, dtype=np.uint8),
                   f"cutoff_{lanes}")
    kw = dict(iter_limit=20, adaptive_step=0, restarts=0, terminate=0, fixed_eta=0.5)
    _, _, r, it = P.pdlp_solve(lp, P.default_params(lanes_A=lanes, lanes_AT=lanes, lanes_kkt_A=lanes,
                                                    lanes_kkt_AT=lanes, **kw), iterates=True)
    ref = O.solve(lp, O.Params(iter_limit=20, adaptive=False, restarts=False, terminate=False, fixed_eta=0.5))
    for k in ("x_cur", "y_cur"):
        want = getattr(ref, k)
        assert np.linalg.norm(it[k] - want) <= 1e-12 * max(1.0, np.linalg.norm(want)), k
    assert abs(r["rel_kkt"] - ref.kkt.rel_kkt) <= 1e-9 * ref.kkt.rel_kkt
