"""Requests with a lifetime cap: the particles' times of flight go through the
shared ring with the request's pass in their sign, in both passes; every tally
equals the single run's."""
import dataclasses

import numpy as np
import pytest

from paper_2503_10263_gb300 import inputs

pytestmark = pytest.mark.gpu

INTEGER = ("spectrum", "time_fx", "cross_pos", "cross_neg", "recomb", "ledger", "chan_count")


@pytest.mark.parametrize("precision", [0, 1])
def test_lifetime_cap_in_a_served_mix(precision):
    from paper_2503_10263_gb300 import karl
    reqs = []
    for i, (n, cap) in enumerate([(1500, 2e-7), (1, 1e-6), (3000, 1e-5), (700, 5e-8), (400, np.inf)]):
        prob, prims = inputs.config2(n, seed=5 + i, column_m2=2e21, nz=150)
        reqs.append((dataclasses.replace(prob, max_lifetime_s=float(cap)), prims))
    srv = karl.Server(reqs[0][0], precision=precision, max_slots=8, hbm_budget_bytes=1 << 29,
                      timeout_s=60)
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
        deaths = got[i]["ledger"][16:48].reshape(4, 8)
        if i != 1:                                          # (one decay may end before its cap)
            assert (deaths[:, 4].sum() > 0) == np.isfinite(p.max_lifetime_s)
