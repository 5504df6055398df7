"""Nearly undamped plates and a nearly undamped shell in FP64 (damping 1e-6 of the usual one): the state
path's factor multiplies by an unevaluated reciprocal pivot above half-bandwidth 8, where beams keep the
correctly rounded one.  Against the oracle; tolerance 1e-9: a long-double integration of such plates puts
either form within 1e-10 of the exact monodromies after 64 steps, the shell's within 1.2e-10, and the
oracle's own rounding is of that size."""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MODELS = {
    "plate_b11": lambda: I.kirchhoff_plate(nx=4, ny=3, n_springs=3, e_count=2, alpha=1e-8, beta=1e-11),
    "plate_b17": lambda: I.kirchhoff_plate(nx=4, ny=5, n_springs=3, e_count=2, alpha=1e-8, beta=1e-11),
    "plate_b35": lambda: I.kirchhoff_plate(nx=3, ny=11, n_springs=3, e_count=2, alpha=1e-8, beta=1e-11),
    "shell": lambda: I.flat_shell(nx=3, ny=5, visc=0.1, zeta1=1e-8),
}


@pytest.mark.parametrize("name", list(MODELS))
def test_nearly_undamped(name):
    from paper_2508_06302_gb300 import fse
    m = MODELS[name]()
    w1 = 1.1 * m.omega_n1
    prob = O.FSEProblem(m, [3], [1], 64, [I.GOLDEN])
    q = np.linalg.solve(m.K + 1j * w1 * m.D - w1 * w1 * m.M, m.F[0])
    C = np.zeros((2 * m.n, prob.U))
    C[:m.n, 0], C[m.n:, 0] = q.real, -q.imag
    C += 1e-3 * np.abs(q).max() * np.random.default_rng(5).standard_normal(C.shape)
    Z = C.reshape(-1)
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=True, dense=False, tol=0, maxit=12)
    with fse.Context(m, 2, [3], [1], [I.GOLDEN], 64, newton_tol=0.0, newton_maxit=12) as ctx:
        R, st, it, rc = ctx.residual_jacobian(Z, w1)
        assert rc == 0
        Phi, dz = ctx.monodromy()
    for a, b in ((R, ref.R), (Phi, ref.Phi), (dz, ref.dz_dw)):
        assert np.linalg.norm(a - b) <= 1e-9 * np.linalg.norm(b)
