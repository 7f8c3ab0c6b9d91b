"""A pass that ends with a primary born below the cutoff, in lanes that take a
parked collision of another request in the same step: every pass end is
published, so every request finishes (long before the launch's deadline) and
equals its single run."""
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


def _request(i, n_dead, n_decays):
    """n_decays decays, then n_dead electrons that are born below the cutoff."""
    prob, pr = inputs.chemistry_config(max(n_decays, 1), 100 + i, column_m2=2e21, nz=40)
    if n_decays == 0:
        pr = pr.slice(0, 0)
    rng = np.random.default_rng(i)
    dead = inputs.Primaries(rng.uniform(0, prob.length_m, n_dead), rng.uniform(0.1, 0.9, n_dead),
                            rng.uniform(-1, 1, n_dead), np.zeros(n_dead, np.uint8), n_dead)
    both = [np.concatenate([getattr(pr, k), getattr(dead, k)])
            for k in ("z_m", "e_ev", "mu", "species")]
    return prob, inputs.Primaries(*both, n_decays + n_dead)


@pytest.mark.parametrize("precision", [0, 1])
def test_passes_that_end_with_a_primary_born_dead(karl, precision):
    # requests of nothing but such primaries among requests whose ions cluster
    # and exchange charge (the collisions that are parked)
    reqs = [_request(i, n_dead=1 + i % 33, n_decays=0 if i % 2 else 1 + i % 7) for i in range(64)]
    ref = []
    for i, (p, q) in enumerate(reqs):
        ctx = karl.Context(p)
        try:
            ref.append(ctx.run(q, seed=50 + i, precision=precision, per_primary=False))
        finally:
            ctx.close()
    for _ in range(12):
        srv = karl.Server(reqs[0][0], precision=precision, max_slots=64, hbm_budget_bytes=1 << 30,
                          timeout_s=20)
        try:
            ids = [srv.submit(p, q, 50 + i) for i, (p, q) in enumerate(reqs)]
            srv.run_all()
            got = [srv.poll(i) for i in ids]
        finally:
            srv.close()
        for i, (done, t) in enumerate(got):
            assert done, i
            for k in INTEGER:
                np.testing.assert_array_equal(t[k], ref[i][k], err_msg=f"{k} of request {i}")
