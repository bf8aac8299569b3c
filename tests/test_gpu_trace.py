"""The decision trace of a float64 solve is that of the solve itself: the same form of the step
kernels, the same point, bit for bit, and decisions that the oracle's replay confirms (check_replay:
iterates to 1e-9 after 150 adaptive, restarted steps, every accept and restart the rule on the
oracle's numbers)."""
import numpy as np
import pytest

import lpgen
from test_gpu_pdlp import P, check_replay  # noqa: F401  (P: the fixture)

pytestmark = pytest.mark.gpu

LPS = {
    "one_block": (lambda: lpgen.mip_relaxation(3, m=60, n=120, density=4 / 60), 3),
    "relaxation": (lambda: lpgen.mip_relaxation(1), 4),
    "cover": (lambda: lpgen.set_cover(7, m=2000, n=8000), 4),
    "energy": (lambda: lpgen.energy_system(hours=24), 4),
}


@pytest.mark.parametrize("name", list(LPS))
def test_recorded_decisions_are_the_solves_own(P, name):  # noqa: F811
    make, form = LPS[name]
    lp = make()
    kw = dict(iter_limit=200, terminate=0)
    x, y, r = P.pdlp_solve(lp, P.default_params(**kw))
    xt, yt, rt, dg = P.pdlp_solve(lp, P.default_params(**kw), trace=2000)
    assert r["persistent_form"] == rt["persistent_form"] == form
    assert r["attempts"] == rt["attempts"] == len(dg["eta"])
    assert np.array_equal(x, xt) and np.array_equal(y, yt)
    assert r["eta"] == rt["eta"] and r["omega"] == rt["omega"]


@pytest.mark.parametrize("name", list(LPS))
def test_replay_of_the_chosen_form(P, name):  # noqa: F811
    check_replay(P, LPS[name][0](), 150)


@pytest.mark.parametrize("name", list(LPS))
def test_replay_with_a_fixed_step(P, name):  # noqa: F811
    """Every attempt accepted; the bound the rule would have used is recorded all the same."""
    lp = LPS[name][0]()
    kw = dict(iter_limit=100, terminate=0, adaptive_step=0, restarts=0, fixed_eta=0.5)
    _, _, r, dg = P.pdlp_solve(lp, P.default_params(**kw), trace=200)
    _, _, r0, dg0 = P.pdlp_solve(lp, P.default_params(lanes_A=2, lanes_AT=2, **kw), trace=200)
    assert (r["persistent_form"], r0["persistent_form"]) == (LPS[name][1], 0)
    assert np.all(dg["accepted"] == 1) and np.all(dg["eta"] == 0.5)
    fin = np.isfinite(dg0["eta_bar"])
    assert np.array_equal(fin, np.isfinite(dg["eta_bar"]))
    np.testing.assert_allclose(dg["eta_bar"][fin], dg0["eta_bar"][fin], rtol=1e-6)
