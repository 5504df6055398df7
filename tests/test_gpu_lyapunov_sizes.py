"""Lyapunov propagation and its QR at the sizes where the kernels change form: cluster sizes 1 to 8
(2n rows), columns at powers of two and next to them, and slices of rows too large for shared memory.
Reference: the oracle's propagation (Householder QR) of the very monodromies the context holds, so the
integration plays no part; tolerance 1e-6 1/s as in test_gpu_parity.py."""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [  # dofs of the chain, samples, exponents, precision
    (1, 1, 1, "fp64"), (3, 3, 5, "fp64"), (8, 5, 16, "mixed_fp32"), (9, 5, 17, "fp64"), (16, 3, 31, "fp64"),
    (33, 5, 33, "mixed_fp32"), (40, 3, 64, "fp64"), (67, 3, 2, "fp64"), (1500, 3, 64, "mixed_fp32"),
    (2100, 3, 64, "fp64"),
]


@pytest.mark.parametrize("n,N,h,precision", CASES)
def test_exponents_of_the_stored_monodromies(n, N, h, precision):
    from paper_2508_06302_gb300 import fse
    m = I.chain(n)
    w1 = 1.15 * max(m.omega_n1, 20.0)
    H = (N - 1) // 2
    ctx = fse.Context(m, 2, [N], [H], [I.GOLDEN], 24, precision=precision)
    ctx.set_steps(24 if n < 1000 else 2)
    Z = I.random_coeffs(m.n, 2 * H + 1, 1e-4, seed=6)
    N_Ly = 12 if n < 1000 else 2
    got = ctx.lyapunov(Z, w1, N_Ly, h)
    prob = O.FSEProblem(m, [N], [H], 24, [I.GOLDEN])
    ref = O.lyapunov(prob, ctx.monodromy()[0], w1, N_Ly=N_Ly, h=h)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-6)
    ctx.close()
