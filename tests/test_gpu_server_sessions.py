"""A closing session goes on publishing waiting requests while the launch finds
nothing left and leaves: each request is then either this launch's, with every
warp of it, or the next one's.  Few slots and many tiny requests, so that the
last one done and the next one published keep meeting; a deadline far below
what a request left behind would wait."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("slots", [1, 2, 5])
def test_requests_published_while_the_launch_leaves(karl, slots, precision):
    reqs = [inputs.config2(1 + i % 3, seed=60 + i, column_m2=5e19, nz=20) for i in range(40)]
    ref = []
    for i, (p, q) in enumerate(reqs):
        ctx = karl.Context(p)
        try:
            ref.append(ctx.run(q, seed=9 + i, precision=precision, per_primary=False))
        finally:
            ctx.close()
    srv = karl.Server(reqs[0][0], precision=precision, max_slots=slots, hbm_budget_bytes=1 << 28,
                      timeout_s=10)
    try:
        for session in range(6):
            ids = [srv.submit(p, q, 9 + i) for i, (p, q) in enumerate(reqs)]
            srv.run_all()
            for i, rid in enumerate(ids):
                done, t = srv.poll(rid)
                assert done, (session, i)
                for k in INTEGER:
                    np.testing.assert_array_equal(t[k], ref[i][k], err_msg=f"{k} of request {i}")
        st = srv.stats()
        assert st.completed == 6 * len(reqs) and st.kernel_launches >= 6
    finally:
        srv.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_a_client_that_only_submits_keeps_its_requests_moving(karl, precision):
    # two slots, a request every 30 ms (several times what one takes), no poll
    # until the end: finished requests make room for waiting ones
    import time
    reqs = [inputs.config2(1 + i % 3, seed=60 + i, column_m2=5e19, nz=20) for i in range(12)]
    srv = karl.Server(reqs[0][0], precision=precision, max_slots=2, hbm_budget_bytes=1 << 28,
                      timeout_s=20)
    try:
        ids = []
        for i, (p, q) in enumerate(reqs):
            ids.append(srv.submit(p, q, 9 + i))
            time.sleep(0.03)
        st = srv.stats()
        srv.run_all()
        got = [srv.poll(i) for i in ids]
    finally:
        srv.close()
    assert st.admitted == len(reqs) and st.waiting == 0 and st.collected == 0
    for i, (done, t) in enumerate(got):
        ctx = karl.Context(reqs[i][0])
        try:
            ref = ctx.run(reqs[i][1], seed=9 + i, precision=precision, per_primary=False)
        finally:
            ctx.close()
        assert done
        for k in INTEGER:
            np.testing.assert_array_equal(t[k], ref[k], err_msg=f"{k} of request {i}")
