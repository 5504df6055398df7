"""Lyapunov exponents called again and again on one context: the QR starts each time from what earlier
launches left in shared memory (norms of other columns, of other sizes), and none of it may reach the
result.  Same reference and tolerance as test_gpu_lyapunov_sizes.py; repeats are equal bit for bit, since
every sum of the propagation has a fixed order."""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,hs", [(3, (5, 1, 6, 2)), (9, (17, 1, 18, 4)), (40, (64, 1, 33, 2))])
def test_exponents_do_not_depend_on_earlier_calls(n, hs):
    from paper_2508_06302_gb300 import fse
    m = I.chain(n)
    w1 = 1.15 * max(m.omega_n1, 20.0)
    prob = O.FSEProblem(m, [3], [1], 24, [I.GOLDEN])
    Z = I.random_coeffs(m.n, 3, 1e-4, seed=6)
    with fse.Context(m, 2, [3], [1], [I.GOLDEN], 24) as ctx:
        first = {}
        for rep in range(4):
            for h in hs:
                got = ctx.lyapunov(Z, w1, 12, h)
                if h not in first:
                    first[h] = got
                    ref = O.lyapunov(prob, ctx.monodromy()[0], w1, N_Ly=12, h=h)
                    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-6)
                assert np.array_equal(got, first[h]), (rep, h)
