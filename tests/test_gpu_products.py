"""J v from the stored monodromies against the same product formed on the host from the monodromies the
context returns (exact copies of what it holds): Eq. 22 in FP64 on both sides, so only the order of the
sums differs.  A dot product of K terms loses at most about K eps of its terms' magnitudes; with
K = 2n + N + U <= 400 and results of the terms' own size, 1e-12 in the 2-norm leaves a factor of ten.
The sizes sit at the edges of the kernels' tiles: 16 rows, vectors of 4, 8 coefficients, 64 samples.
"""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = {
    "chain1": (lambda: I.chain(1), 1, 0, 1),
    "chain8_N64": (lambda: I.chain(8), 64, 3, 2),
    "chain17_N65": (lambda: I.chain(17), 65, 4, 3),
    "chain64_decay": (lambda: I.chain(64), 5, 2, 4),   # far entries underflow in FP32
    "plate27": (lambda: I.kirchhoff_plate(nx=4, ny=4, n_springs=3, e_count=2), 9, 4, 5),
    "shell90": (lambda: I.flat_shell(nx=6, ny=4), 7, 3, 1),
    "plate114_pipelined": (lambda: I.kirchhoff_plate(nx=3, ny=20, n_springs=3, e_count=2), 151, 75, 3),
}


@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("name", list(CASES))
def test_products_from_stored_monodromies(name, precision):
    from paper_2508_06302_gb300 import fse
    mk, N, H, nvec = CASES[name]
    m = mk()
    w1 = 1.1 * m.omega_n1
    prob = O.FSEProblem(m, [N], [H], 24, [I.GOLDEN])
    ctx = fse.Context(m, 2, [N], [H], [I.GOLDEN], 24, precision=precision)
    ctx.set_steps(3)
    ctx.residual_jacobian(I.random_coeffs(m.n, prob.U, 1e-4, seed=2), w1)
    Phi = ctx.monodromy()[0]
    V = np.random.default_rng(4).standard_normal((nvec, 2 * m.n * prob.U))
    got = ctx.jacobian_apply(V)
    RG = prob.R @ prob.Gi
    for k in range(nvec):
        v = V[k].reshape(2 * m.n, prob.U)
        want = (RG @ np.einsum("sij,sj->si", Phi, prob.G @ v.T)).T - v
        assert np.linalg.norm(got[k].reshape(want.shape) - want) <= 1e-12 * np.linalg.norm(want)
    ctx.close()
