"""J v and the DFT in every form the sizes choose: rows in groups of 16 or 32 lanes, rows of a dof in pairs,
the staged FP32 form, with one panel and with several; the DFT with its lanes over the samples and with 4 and
8 warps to a tile, at the edges of the rules.  Reference and tolerance as in test_gpu_products.py (FP64 on
both sides from the very monodromies the context holds, K <= 1800 terms of size one: K eps = 4e-13)."""
import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def blocks(*sizes):
    """Independent chains one after the other: a panel each (the small ones share one)."""
    parts = [I.chain(k) for k in sizes]
    n, o = sum(sizes), 0
    M, D, K = np.zeros((n, n)), np.zeros((n, n)), np.zeros((n, n))
    dofs = []
    for k, p in zip(sizes, parts):
        s = slice(o, o + k)
        M[s, s], D[s, s], K[s, s] = p.M, p.D, p.K
        dofs.append(np.where(p.nl_dof >= 0, p.nl_dof + o, -1))
        o += k
    F = np.zeros((2, n))
    F[:, 0] = 1.0, 0.5
    return I.FEModel("blocks", M, D, K, np.concatenate([p.nl_type for p in parts]).astype(np.int32),
                     np.concatenate(dofs).astype(np.int32), np.concatenate([p.nl_p for p in parts]), F,
                     min(p.omega_n1 for p in parts))


CASES = [  # model, samples, harmonics, precision
    (lambda: I.chain(1), 1, 0, "fp64"), (lambda: I.chain(6), 63, 31, "fp64"),                  # 32 lanes
    (lambda: I.chain(64), 8, 3, "fp64"), (lambda: I.chain(256), 3, 1, "fp64"),                 # 16 lanes
    (lambda: I.chain(257), 3, 1, "fp64"), (lambda: I.chain(257), 9, 4, "fp64"),                # 32 lanes; pairs
    (lambda: I.chain(301), 17, 8, "fp64"),
    (lambda: blocks(40, 33), 5, 2, "fp64"), (lambda: blocks(100, 70, 9, 2), 9, 4, "fp64"),
    (lambda: blocks(290, 150, 50), 9, 4, "fp64"),
    (lambda: I.chain(1), 1, 0, "mixed_fp32"), (lambda: I.chain(128), 5, 2, "mixed_fp32"),      # 32; 16 lanes
    (lambda: I.chain(129), 5, 2, "mixed_fp32"), (lambda: I.chain(153), 16, 7, "mixed_fp32"),   # 32 lanes; 1.498 M
    (lambda: I.chain(154), 16, 7, "mixed_fp32"), (lambda: I.chain(578), 3, 1, "mixed_fp32"),   # staged
    (lambda: blocks(60, 40), 7, 3, "mixed_fp32"), (lambda: blocks(240, 150, 9, 2), 9, 4, "mixed_fp32"),
    # DFT: lanes over the samples up to 23 states, 47 with at most 32 samples and, with many samples, beyond;
    # tiles of 32 states, four warps each up to 16 samples or with many tiles, else eight
    (lambda: I.chain(11), 40, 19, "fp64"), (lambda: I.chain(12), 40, 19, "fp64"), (lambda: I.chain(18), 225, 112, "fp64"),
    (lambda: I.chain(16), 9, 4, "fp64"), (lambda: I.chain(17), 9, 4, "fp64"), (lambda: I.chain(63), 131, 65, "fp64"),
    (lambda: I.chain(64), 131, 65, "fp64"), (lambda: I.chain(50), 2, 0, "fp64"),
    (lambda: I.chain(23), 32, 15, "fp64"), (lambda: I.chain(23), 33, 16, "fp64"), (lambda: I.chain(24), 32, 15, "fp64"),
    (lambda: I.chain(24), 16, 7, "fp64"), (lambda: I.chain(24), 17, 8, "fp64"), (lambda: I.chain(33), 7, 3, "fp64"),
]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_product_forms(k):
    from paper_2508_06302_gb300 import fse
    mk, N, H, precision = CASES[k]
    m = mk()
    w1 = 1.1 * m.omega_n1
    prob = O.FSEProblem(m, [N], [H], 24, [I.GOLDEN])
    with fse.Context(m, 2, [N], [H], [I.GOLDEN], 24, precision=precision) as ctx:
        ctx.set_steps(3)
        ctx.residual_jacobian(I.random_coeffs(m.n, prob.U, 1e-4, seed=2), w1)
        Phi, dz = ctx.monodromy()
        V = np.random.default_rng(4).standard_normal((2, 2 * m.n * prob.U))
        got, dw = ctx.jacobian_apply(V), ctx.jacobian_domega()
    RG = prob.R @ prob.Gi

    def close(a, b):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)

    for v, g in zip(V, got):
        v = v.reshape(2 * m.n, prob.U)
        close(g.reshape(v.shape), (RG @ np.einsum("sij,sj->si", Phi, prob.G @ v.T)).T - v)
    close(dw.reshape(2 * m.n, prob.U), (RG @ dz).T)
