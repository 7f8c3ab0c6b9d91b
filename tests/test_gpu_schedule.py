"""Which warp follows a particle changes no tally: runs of few primaries (an
equal share per scheduler), of more than one warp per scheduler holds, and of
more than the chip holds, against the same runs in one- and three-warp blocks,
every integer tally bit for bit."""
import numpy as np
import pytest

from paper_2503_10263_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def karl():
    from paper_2503_10263_gb300 import karl as k
    k.load()
    return k


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_decays", [1, 303, 304, 305, 9729, 45000])
def test_tallies_do_not_depend_on_the_launch_shape(karl, n_decays, precision):
    prob, prims = inputs.config2(n_decays, seed=11, column_m2=6e20, nz=64)
    ctx = karl.Context(prob)
    try:
        a = ctx.run(prims, seed=3, precision=precision)
        b = ctx.run(prims, seed=3, precision=precision, block_size=96, blocks_per_sm=2)
        c = ctx.run(prims, seed=3, precision=precision, block_size=32, blocks_per_sm=1)
    finally:
        ctx.close()
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
        np.testing.assert_array_equal(a[k], c[k], err_msg=k)
    L = a["ledger"]
    assert L[karl.E_IN_PRIMARY] + L[karl.E_IN_THERMAL] == L[karl.E_EXIT0:karl.E_STALLED + 1].sum()
