"""The sums along z, the target fields and the normalisation after a pass at
sizes around their kernels' cuts (32 columns, 32 stretches of rows, 128 energy
bins, 256 segments of a column), against the oracle on histories that match it
and against plain sums of the same run's tallies."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2503_10263_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def karl():
    from paper_2503_10263_gb300 import karl as k
    k.load()
    return k


@pytest.mark.parametrize("nz,ntb", [(1, 1), (2, 3), (30, 8), (31, 129), (257, 64), (1025, 7)])
def test_tallies_along_z(karl, nz, ntb):
    prob, prims = inputs.config2(40, seed=3, column_m2=5e19, nz=nz)
    prob = dataclasses.replace(prob, n_tebins=ntb)
    ctx = karl.Context(prob)
    try:
        g = ctx.run(prims, seed=2)
        c = ctx.run_cycles(prims, 2, 2)
    finally:
        ctx.close()
    o = oracle.run(prob, prims, seed=2, n_threads=4)
    np.testing.assert_array_equal(g["per_primary"], o["per_primary"])
    for k in ("cross_pos", "cross_neg", "recomb"):
        np.testing.assert_array_equal(g[k], o[k], err_msg=k)
    # the kernel's time quanta are the oracle's to one unit per segment visit
    visits = 4.0 * (o["cross_pos"].sum() + o["cross_neg"].sum() + o["ledger"][karl.N_FLIGHTS])
    assert abs(float(g["time_fx"].sum()) - float(o["time_fx"].sum())) <= visits
    for k in ("density", "current", "field"):
        scale = max(np.abs(o[k]).max(), 1e-300)
        np.testing.assert_allclose(g[k] / scale, o[k] / scale, rtol=0, atol=1e-6, err_msg=k)
    # normalisation of this run's own tallies (two cycles: fields with deletions)
    tsim, vol = prims.n_decays / prob.activity_bq, prob.length_m / nz * prob.area_m2
    for t in (g, c):
        sec = t["time_fx"][:, 1:nz + 1, :].astype(float).sum(axis=2) / 2.0 ** 50
        want = sec / (tsim * vol) - t["recomb"].astype(float) / vol
        np.testing.assert_allclose(t["density"], want, rtol=1e-12,
                                   atol=1e-12 * np.abs(want).max())
        cur = (t["cross_pos"].astype(float) - t["cross_neg"].astype(float)) / (prob.area_m2 * tsim)
        np.testing.assert_allclose(t["current"], cur, rtol=1e-14)
