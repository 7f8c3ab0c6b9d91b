"""The work between a request's passes is cut into units of 32 segments or 32
(species, energy bin) columns that any warp takes; at sizes around those cuts,
and with several requests between passes at once, every tally equals the
single-run path's."""
import dataclasses

import numpy as np
import pytest

from paper_2503_10263_gb300 import inputs

pytestmark = pytest.mark.gpu

INTEGER = ("spectrum", "time_fx", "cross_pos", "cross_neg", "recomb", "ledger", "chan_count")


@pytest.fixture(scope="module")
def karl():
    from paper_2503_10263_gb300 import karl as k
    k.load()
    return k


def _source(n, nz, ntb, seed):
    prob, prims = inputs.config2(n, seed=seed, column_m2=4e20, nz=nz)
    return dataclasses.replace(prob, n_tebins=ntb), prims


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nz,ntb", [(1, 1), (8, 9), (31, 33), (32, 64), (33, 5), (257, 64)])
def test_units_at_their_edges(karl, nz, ntb, precision):
    reqs = [_source(n, nz, ntb, 5 + i) for i, n in enumerate((1, 40, 700, 1500))]
    srv = karl.Server(reqs[0][0], precision=precision, max_slots=8, hbm_budget_bytes=1 << 29)
    try:
        ids = [srv.submit(p, q, 17 + i) for i, (p, q) in enumerate(reqs)]
        srv.run_all()
        got = [srv.poll(i)[1] for i in ids]
    finally:
        srv.close()
    for i, (p, q) in enumerate(reqs):
        ctx = karl.Context(p)
        try:
            ref = ctx.run(q, seed=17 + i, precision=precision)
        finally:
            ctx.close()
        for k in INTEGER:
            np.testing.assert_array_equal(got[i][k], ref[k], err_msg=f"{k} of request {i}")
        for k in ("density", "current", "field"):
            np.testing.assert_allclose(got[i][k], ref[k], rtol=1e-12, err_msg=k)
