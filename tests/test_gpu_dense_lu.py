"""Dense outer solve at the sizes where the blocked LU changes form: fewer unknowns than a panel of 16
columns, one panel, ragged last panels and 64-wide tiles, and panels too long for shared memory (beyond
1500 rows).  The Newton update against numpy's solve of the Jacobian the context returns; 1e-8 relative as
for the dense update in test_gpu_gmres.py."""
import numpy as np
import pytest

from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H", [(1, 0), (4, 0), (8, 0), (3, 1), (11, 1), (13, 2), (51, 7)])
def test_newton_update_equals_dense_solve(n, H):
    from paper_2508_06302_gb300 import fse
    m = I.chain(n, c=30.0)
    w1 = 1.1 * max(m.omega_n1, 20.0)
    N = 2 * H + 1
    ctx = fse.Context(m, 2, [N], [H], [I.GOLDEN], 16, newton_tol=0.0, newton_maxit=8)
    ctx.set_linear_solver("dense")
    Z = I.random_coeffs(m.n, N, 1e-4, seed=8)
    R, st, it, rc = ctx.residual_jacobian(Z, w1)
    want = np.linalg.solve(ctx.jacobian_dense(), -R)
    Zn, rn, rc = ctx.newton_step(Z, w1)
    assert rc == 0 and abs(rn - np.linalg.norm(R)) <= 1e-12 * rn
    assert np.linalg.norm(Zn - Z - want) <= 1e-8 * np.linalg.norm(want)
    ctx.close()
