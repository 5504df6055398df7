"""Column Cholesky at half-bandwidths where a column has rows in more than one warp (32 and more): the
mass factor behind the start acceleration, and the FP32 factor of undivided models beyond the panel factor
(half-bandwidth 98).  One Newmark step shows the start acceleration at full size.  Tolerance 1e-12 of
|Z| + |R| (start acceleration, one step and the DFT in FP64 on both sides, a few hundred roundings of 1e-16
each, the mass matrix scaled by its own diagonal well conditioned); repeats, the factor formed anew by each
context, are equal bit for bit."""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,band,precision", [(9, 29, "fp64"), (10, 32, "fp64"), (11, 35, "fp64"), (31, 95, "mixed_fp32")])
def test_start_acceleration(ny, band, precision):
    from paper_2508_06302_gb300 import fse
    m = I.kirchhoff_plate(nx=4, ny=ny, n_springs=3, e_count=2)
    w1 = 1.1 * m.omega_n1
    prob = O.FSEProblem(m, [5], [2], 200, [I.GOLDEN])
    Z = I.random_coeffs(m.n, 5, 1e-5, seed=7)
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=False, tol=0, maxit=8, n_steps=1).R
    first = None
    for rep in range(6):
        with fse.Context(m, 2, [5], [2], [I.GOLDEN], 200, newton_tol=0.0, newton_maxit=8, precision=precision) as ctx:
            assert ctx.band == band
            ctx.set_steps(1)
            R, st, it, rc = ctx.residual_jacobian(Z, w1, want_jacobian=False)
        assert rc == 0
        assert np.linalg.norm(R - ref) <= 1e-12 * (np.linalg.norm(Z) + np.linalg.norm(ref))
        first = R if first is None else first
        assert np.array_equal(R, first), rep


def test_wide_fp32_factor_repeats():
    from paper_2508_06302_gb300 import fse
    m = I.kirchhoff_plate(nx=4, ny=32, n_springs=3, e_count=2)
    w1 = 1.1 * m.omega_n1
    Z = I.random_coeffs(m.n, 5, 1e-5, seed=7)
    with fse.Context(m, 2, [5], [2], [I.GOLDEN], 200, newton_tol=0.0, newton_maxit=8, precision="mixed_fp32") as ctx:
        assert ctx.band == 98
        ctx.set_steps(6)
        first = None
        for rep in range(6):
            assert ctx.residual_jacobian(Z, w1)[3] == 0
            Phi = ctx.monodromy()[0]
            first = Phi if first is None else first
            assert np.array_equal(Phi, first), rep
