"""The exchange of the resident step kernel (persistent_form 4): LPs whose blocks need nothing of one
another but the sums, so that they run as far apart as the exchange allows.

Tolerances as in test_gpu_resident: a few hundred roundings after 60 fixed steps."""
import numpy as np
import pytest

import lpgen
from test_gpu_resident import F32, F64, FIXED, P, rel  # noqa: F401  (P: the fixture)

pytestmark = pytest.mark.gpu


def uncoupled(pieces, size=8, seed=1):
    """Independent dense pieces of size x size."""
    rng = np.random.default_rng(seed)
    m = pieces * size
    rows = np.repeat(np.arange(m), size)
    cols = (rows // size) * size + np.tile(np.arange(size), m)
    return lpgen._lp(m, m, rows, cols, rng.integers(1, 4, rows.size).astype(float), rng.uniform(0, 2, m),
                     rng.choice([lpgen.SENSE_GE, lpgen.SENSE_EQ], m), rng.uniform(-1, 1, m),
                     np.zeros(m), rng.uniform(1, 5, m), np.zeros(m, dtype=np.uint8), f"pieces_{pieces}")


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("pieces", [60, 400, 1600])  # a few blocks, about a hundred, every SM
def test_uncoupled_blocks(P, pieces, prec):  # noqa: F811
    lp = uncoupled(pieces)
    tol = F64 if prec == "fp64" else F32
    x, y, r = P.pdlp_solve(lp, P.default_params(precision=prec, **FIXED))
    x0, y0, r0 = P.pdlp_solve(lp, P.default_params(precision=prec, lanes_A=2, lanes_AT=2, **FIXED))
    assert r["persistent_form"] == 4 and r0["persistent_form"] == 0
    assert rel(x, x0) <= tol and rel(y, y0) <= tol
    _, _, r = P.pdlp_solve(lp, P.default_params(precision=prec, **dict(FIXED, iter_limit=20000)))
    assert r["persistent_form"] == 4 and r["iters"] == 20000


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("name", ["cover", "uncoupled"])
def test_withheld_sums_time_out_and_the_context_survives(P, name, prec):  # noqa: F811
    """Block 0 begins only when another block's bounded wait has run out (for its entries, or where the
    blocks are not coupled for its sums): every block leaves, the call reports PDLP_ERR_TIMEOUT, and
    the next solve in the same form succeeds."""
    lp = lpgen.set_cover(7, m=2000, n=8000) if name == "cover" else uncoupled(400)
    with pytest.raises(P.PdlpError, match="PDLP_ERR_TIMEOUT"):
        P.pdlp_solve(lp, P.default_params(precision=prec, debug_skip_barrier=1))
    _, _, r = P.pdlp_solve(lp, P.default_params(precision=prec, iter_limit=200, terminate=0))
    assert r["persistent_form"] == 4 and r["iters"] == 200


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", ["cover", "uncoupled"])
def test_a_late_block_that_completes_its_attempt_still_fails_the_solve(P, name, prec):  # noqa: F811
    """With one attempt per check period the late block 0 finds all that it needs where the blocks
    are not coupled, and leaves as after a success, while the others have left without their part
    of the iterate."""
    lp = lpgen.set_cover(7, m=2000, n=8000) if name == "cover" else uncoupled(400)
    kw = dict(precision=prec, adaptive_step=0, check_period=1)
    with pytest.raises(P.PdlpError, match="PDLP_ERR_TIMEOUT"):
        P.pdlp_solve(lp, P.default_params(debug_skip_barrier=1, iter_limit=50, **kw))
    with pytest.raises(P.PdlpError, match="PDLP_ERR_TIMEOUT"):
        P.pdlp_solve(lp, P.default_params(debug_skip_barrier=1, iter_limit=1, **kw))
    _, _, r = P.pdlp_solve(lp, P.default_params(iter_limit=50, terminate=0, **kw))
    assert r["persistent_form"] == 4 and r["iters"] == 50
