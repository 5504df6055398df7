"""FP64 tangents of undivided plates across the half-bandwidths at which the row-by-row solves change
their register window (4, 8, 16, 24, 32) and give way to the blocked solves (b = 35), with row counts
around the 32-row chunks and the groups of four rows; against the oracle, 1e-10 relative as in
test_gpu_parity.py."""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (4, 2), (12, 2), (3, 3), (3, 4), (5, 7), (4, 8), (3, 10), (3, 11)])
def test_plate_monodromies_fp64(nx, ny):
    from paper_2508_06302_gb300 import fse
    m = I.kirchhoff_plate(nx=nx, ny=ny, n_springs=1, e_count=2)
    w1 = 1.1 * m.omega_n1
    prob = O.FSEProblem(m, [3], [1], 10, [I.GOLDEN])
    Z = I.random_coeffs(m.n, 3, 1e-4, seed=9)
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=True, dense=False, tol=0, maxit=10)
    ctx = fse.Context(m, 2, [3], [1], [I.GOLDEN], 10, newton_tol=0.0, newton_maxit=10)
    R, st, it, rc = ctx.residual_jacobian(Z, w1)
    assert rc == 0
    Phi, dz = ctx.monodromy()
    for a, b in ((R, ref.R), (Phi, ref.Phi), (dz, ref.dz_dw)):
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
    ctx.close()
