"""The separate launches (persistent_form 0), asked for by their lanes, against every other form of
the step kernels: with persistent = 0 alone a single LP that fits takes another form.  After 60
fixed steps the iterates agree to a few hundred roundings, and solved to 1e-4 the point passes the
oracle's float64 KKT."""
import pytest

import lpgen
from oracle import pdlp_oracle as O
from test_gpu_resident import F32, F64, FIXED, P, rel  # noqa: F401  (P: the fixture)

pytestmark = pytest.mark.gpu

LPS = {
    "relaxation": lambda: lpgen.mip_relaxation(1),
    "free_and_eq": lambda: lpgen.random_sparse_lp(11, 300, 500),
    "cover": lambda: lpgen.set_cover(7, m=300, n=1200),
}
OTHERS = [dict(persistent=1), dict(persistent=2), dict(tiles=1), dict(tiles=2), dict()]


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("lanes", [(1, 1), (2, 2), (8, 4)])
@pytest.mark.parametrize("name", list(LPS))
def test_launches_agree_with_the_other_forms(P, name, lanes, prec):  # noqa: F811
    lp = LPS[name]()
    tol = F64 if prec == "fp64" else F32
    ref = O.solve(lp, O.Params(iter_limit=60, adaptive=False, restarts=False, terminate=False,
                               fixed_eta=0.9))
    x0, y0, r0, it0 = P.pdlp_solve(lp, P.default_params(precision=prec, lanes_A=lanes[0],
                                                        lanes_AT=lanes[1], **FIXED), iterates=True)
    assert r0["persistent_form"] == 0 and r0["tiles"] == 0 and r0["iters"] == 60
    for k in ("x_cur", "y_cur", "x_avg", "y_avg"):
        assert rel(it0[k], getattr(ref, k)) <= tol, (k, rel(it0[k], getattr(ref, k)))
    for kw in OTHERS:
        if "tiles" in kw and prec == "fp64":
            continue
        x, y, r = P.pdlp_solve(lp, P.default_params(precision=prec, **kw, **FIXED))
        assert r["tiles"] == kw.get("tiles", 0)
        if "tiles" not in kw:
            assert r["persistent_form"] > 0, (kw, r["persistent_form"])
        assert rel(x, x0) <= tol and rel(y, y0) <= tol, (kw, rel(x, x0), rel(y, y0))


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("lanes", [(1, 1), (4, 2)])
@pytest.mark.parametrize("name", list(LPS))
def test_launches_reach_the_tolerance(P, name, lanes, prec):  # noqa: F811
    lp = LPS[name]()
    x, y, r = P.pdlp_solve(lp, P.default_params(tol=1e-4, precision=prec, lanes_A=lanes[0],
                                                lanes_AT=lanes[1]))
    assert r["status"] == P.PDLP_OPTIMAL and r["persistent_form"] == 0
    assert (r["lanes_A"], r["lanes_AT"]) == lanes
    assert O.kkt_original(lp, x, y).rel_kkt <= 1.01e-4


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_one_block_up_to_where_it_is_faster(P, prec):  # noqa: F811
    def form(lp):
        return P.pdlp_solve(lp, P.default_params(iter_limit=5, terminate=0, precision=prec))[2]["persistent_form"]

    assert form(lpgen.set_cover(1, m=100, n=400)) == 3                              # 2,668 nonzeros
    assert form(lpgen.mip_relaxation(1, m=300, n=600)) == 3                         # 3,642
    assert form(lpgen.mip_relaxation(1, m=600, n=1200, density=4 / 600)) == 4       # 4,843
    assert form(lpgen.random_sparse_lp(1, 20, 1500, density=0.1)) == 4              # 3,000, long rows
