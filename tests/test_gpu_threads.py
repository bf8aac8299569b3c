"""More solves at once than the cache of captured graphs has entries (8): a graph that a solve of
another thread still launches stays."""
import threading

import numpy as np
import pytest

import lpgen
from test_gpu_resident import P  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

THREADS = 12


@pytest.mark.parametrize("kw", [dict(precision="bf16"), dict(precision="fp64", lanes_A=2, lanes_AT=2)])
def test_more_solves_at_once_than_cached_graphs(P, kw):  # noqa: F811
    lps = [lpgen.mip_relaxation(s, m=200 + 10 * s, n=400 + 20 * s) for s in range(THREADS)]
    prm = dict(kw, iter_limit=256, terminate=0)
    alone = [P.pdlp_solve(lp, P.default_params(**prm)) for lp in lps]
    got, failed = [[] for _ in lps], []

    def work(k):
        try:
            for _ in range(4):
                got[k].append(P.pdlp_solve(lps[k], P.default_params(**prm)))
        except P.PdlpError as e:
            failed.append((k, str(e)))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(THREADS)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed
    for k in range(THREADS):
        for x, y, r in got[k]:
            assert np.array_equal(x, alone[k][0]) and np.array_equal(y, alone[k][1])
            assert r["kernel_launches"] == alone[k][2]["kernel_launches"]
