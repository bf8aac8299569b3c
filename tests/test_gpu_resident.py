"""The resident step kernel (persistent_form 4: one LP spread over the SMs' shared memory) and the
rule that chooses it.

Iterates after 60 fixed steps agree with the float64 oracle's and with the separate launches' to
rounding (a few hundred roundings: of 6e-8 in float32, 2e-5 as for the other forms; of 1.1e-16 in
float64, 1e-12).  The sizes put
rows and columns at the lengths where a warp takes over (64, 65), parts into several stages, and
blocks without rows.
"""
import threading

import numpy as np
import pytest

import lpgen
from oracle import pdlp_oracle as O

pytestmark = pytest.mark.gpu

F32, F64 = 2e-5, 1e-12
FIXED = dict(adaptive_step=0, restarts=0, terminate=0, fixed_eta=0.9, iter_limit=60)


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as G
    G.build()
    import paper_2503_10344_gb300 as P
    return P


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(1.0, np.linalg.norm(b)))


def rows_of(lengths, n, seed):
    """Rows of the given lengths over n columns, mixed senses, small integer values."""
    rng = np.random.default_rng(seed)
    m = len(lengths)
    rows = np.repeat(np.arange(m), lengths)
    cols = np.concatenate([rng.choice(n, k, replace=False) for k in lengths])
    val = rng.integers(1, 4, rows.size) * rng.choice([-1.0, 1.0], rows.size)
    return lpgen._lp(m, n, rows, cols, val, rng.uniform(0, 2, m),
                     rng.choice([lpgen.SENSE_GE, lpgen.SENSE_LE, lpgen.SENSE_EQ], m),
                     rng.uniform(-1, 1, n), np.zeros(n), rng.uniform(1, 5, n),
                     np.zeros(n, dtype=np.uint8), f"rows_{m}x{n}")


LPS = {
    "threshold_rows": lambda: rows_of([64, 65, 1, 2, 63] * 20, 700, 1),
    "one_long_row": lambda: rows_of([6000] + [1] * 40, 6001, 2),
    "few_rows": lambda: rows_of([1500, 1600], 2000, 3),
    "empty_rows_and_columns": lambda: rows_of(([0] * 7 + [9]) * 300, 9000, 4),
    "some_empty_rows_and_columns": lambda: rows_of(([0] * 3 + [19]) * 200, 2500, 6),
    "odd_cover": lambda: lpgen.set_cover(3, m=1777, n=7103),
    "skewed": lpgen.skewed_lp,
    "energy_31h": lambda: lpgen.energy_system(hours=31),
}

# vectors that do not fit in the scratch the setup leaves (the workspace does not grow for them):
# the separate launches run
NOT_RESIDENT = {"empty_rows_and_columns"}
NOT_RESIDENT_F64 = NOT_RESIDENT | {"one_long_row", "some_empty_rows_and_columns"}  # (twice the size)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name", list(LPS))
def test_resident_iterates(P, name, prec):
    lp = LPS[name]()
    _, _, r, it = P.pdlp_solve(lp, P.default_params(precision=prec, **FIXED), iterates=True)
    _, _, r0, it0 = P.pdlp_solve(lp, P.default_params(precision=prec, lanes_A=2, lanes_AT=2, **FIXED),
                                 iterates=True)
    assert r["persistent_form"] == (0 if name in NOT_RESIDENT else 4)
    assert r0["persistent_form"] == 0
    assert r["iters"] == r0["iters"] == 60
    ref = O.solve(lp, O.Params(iter_limit=60, adaptive=False, restarts=False, terminate=False,
                               fixed_eta=0.9))
    for k in ("x_cur", "y_cur", "x_avg", "y_avg"):
        assert rel(it[k], it0[k]) <= F32, (k, rel(it[k], it0[k]))
        assert rel(it[k], getattr(ref, k)) <= F32, (k, rel(it[k], getattr(ref, k)))


@pytest.mark.parametrize("name", list(LPS))
def test_resident_float64(P, name):
    """(A solve that records iterates keeps the separate launches: the points are compared.)"""
    lp = LPS[name]()
    x, y, r = P.pdlp_solve(lp, P.default_params(**FIXED))
    x0, y0, r0 = P.pdlp_solve(lp, P.default_params(lanes_A=2, lanes_AT=2, **FIXED))
    assert r["persistent_form"] == (0 if name in NOT_RESIDENT_F64 else 4)
    assert r0["persistent_form"] == 0
    assert P.pdlp_solve(lp, P.default_params(**FIXED), iterates=True)[2]["persistent_form"] == 0
    ref = O.solve(lp, O.Params(iter_limit=60, adaptive=False, restarts=False, terminate=False,
                               fixed_eta=0.9))
    for got, want in ((x, x0), (y, y0), (x, ref.x), (y, ref.y)):
        assert rel(got, want) <= F64, rel(got, want)


def test_several_stages(P):
    """The 50,000 x 200,000 covering LP with float32 values: the entries of a part are staged
    in more than one go."""
    lp = lpgen.set_cover(2025)
    kw = dict(FIXED, iter_limit=20)
    _, _, r, it = P.pdlp_solve(lp, P.default_params(precision="fp32", **kw), iterates=True)
    _, _, _, it0 = P.pdlp_solve(lp, P.default_params(precision="fp32", lanes_A=8, lanes_AT=1, **kw),
                                iterates=True)
    assert r["persistent_form"] == 4
    for k in ("x_cur", "y_cur", "x_avg", "y_avg"):
        assert rel(it[k], it0[k]) <= F32, (k, rel(it[k], it0[k]))


def test_float64_values_from_global_memory(P):
    """A part of the LP with its stage is more than an SM holds: the float64 values stay in global
    memory and are staged, with the entries they multiply, in several goes."""
    lp = lpgen.set_cover(9, m=36000, n=144000)
    kw = dict(FIXED, iter_limit=20)
    x, y, r = P.pdlp_solve(lp, P.default_params(**kw))
    x0, y0, r0 = P.pdlp_solve(lp, P.default_params(lanes_A=8, lanes_AT=2, **kw))
    assert r["persistent_form"] == 4 and r0["persistent_form"] == 0
    assert rel(x, x0) <= F64 and rel(y, y0) <= F64


def test_rejected_steps_float64(P):
    """As below; a rounding grows about tenfold every 40 adaptive steps, 1e-9 after 100."""
    lp = lpgen.set_cover(5, m=1500, n=6000)
    prm = dict(fixed_eta=200.0, iter_limit=100, terminate=0)
    x, y, r = P.pdlp_solve(lp, P.default_params(**prm))
    x0, y0, r0 = P.pdlp_solve(lp, P.default_params(lanes_A=2, lanes_AT=2, **prm))
    assert r["persistent_form"] == 4 and r0["persistent_form"] == 0
    assert r["attempts"] == r0["attempts"] > r["iters"] == 100
    assert rel(x, x0) <= 1e-9 and rel(y, y0) <= 1e-9


def test_rejected_steps(P):
    """A start step far above the bound: rejected attempts read the kept y again.  Every decision
    follows the rule, and the solve ends at the tolerance."""
    lp = lpgen.set_cover(5, m=1500, n=6000)
    prm = dict(precision="bf16", fixed_eta=200.0)
    _, _, r, dg = P.pdlp_solve(lp, P.default_params(iter_limit=128, terminate=0, **prm), trace=2000)
    assert r["persistent_form"] == 4 and r["attempts"] > r["iters"] == 128
    assert np.array_equal(dg["accepted"] == 1, ~(dg["eta"] > dg["eta_bar"]))
    x, y, r = P.pdlp_solve(lp, P.default_params(tol=1e-4, **prm))
    assert r["status"] == P.PDLP_OPTIMAL and O.kkt_original(lp, x, y).rel_kkt <= 1.01e-4


def test_form_by_size(P):
    def form(lp, **kw):
        return P.pdlp_solve(lp, P.default_params(iter_limit=5, terminate=0, **kw))[2]["persistent_form"]

    small, mid = lpgen.mip_relaxation(1), lpgen.set_cover(7, m=2000, n=8000)
    assert form(small, precision="fp32") == 3 and form(mid, precision="fp32") == 4
    assert form(small, precision="fp64") == form(mid, precision="fp64") == 4
    assert form(lpgen.mip_relaxation(3, m=60, n=120, density=4 / 60), precision="fp64") == 3
    assert form(lpgen.set_cover(2025), precision="fp64") == 0  # more than the SMs hold
    for kw in (dict(precision="fp64", lanes_A=2), dict(precision="fp32", lanes_A=2), dict(precision="bf16", autotune=1),
               dict(precision="fp32", tiles=1), dict(precision="fp32", halpern=1)):
        assert form(small, **kw) == form(mid, **kw) == 0, kw
    assert form(lpgen.energy_system(hours=2880), precision="fp32") == 0  # more than the SMs hold


def test_two_threads_at_once(P):
    """Solves of two host threads, each large enough to ask for every SM, give the bits of solves
    run alone."""
    lps = [lpgen.set_cover(11, m=12000, n=48000), lpgen.set_cover(12, m=9000, n=36000)]
    prm = dict(precision="bf16", iter_limit=256, terminate=0)
    alone = [P.pdlp_solve(lp, P.default_params(**prm)) for lp in lps]
    assert all(a[2]["persistent_form"] == 4 for a in alone)
    got = [[], []]

    def work(k):
        for _ in range(4):
            got[k].append(P.pdlp_solve(lps[k], P.default_params(**prm)))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for k in range(2):
        assert len(got[k]) == 4
        for x, y, _ in got[k]:
            assert np.array_equal(x, alone[k][0]) and np.array_equal(y, alone[k][1])
