"""Models whose dofs divide into panels, in what reads them beyond the calls of test_gpu_panels.py: batches
(on streams and as one captured graph), trajectory shards, and the bordered Newton update of an unknown base
frequency.  Batches equal the evaluations one by one bit for bit (test_gpu_batch.py), shard sums agree to
1e-13 (test_gpu_shard.py), the update to the oracle's within 1e-8 as the dense update there."""
import numpy as np
import pytest

from oracle import unknown_freq as UF
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def two_chains(a, b, vdp=False):
    """Two chains that nothing couples, their dofs alternating; vdp: a self-excited damper on the second."""
    n = a + b
    order = np.argsort(np.concatenate([(np.arange(a) + 0.5) / a, (np.arange(b) + 0.5) / b]), kind="stable")
    pos = np.empty(n, int)
    pos[order] = np.arange(n)   # chain dof -> dof of the model
    M, D, K = (np.zeros((n, n)) for _ in range(3))
    typ, dof, par = [], [], []
    for o, p in ((0, I.chain(a)), (a, I.chain(b, k=1.3e4))):
        ix = pos[o:o + p.n]
        M[np.ix_(ix, ix)], D[np.ix_(ix, ix)], K[np.ix_(ix, ix)] = p.M, p.D, p.K
        typ.append(p.nl_type)
        dof.append(np.where(p.nl_dof >= 0, ix[np.maximum(p.nl_dof, 0)], -1))
        par.append(p.nl_p)
    if vdp:
        typ.append([I.NL_VDP])
        dof.append([[pos[a], -1, -1, -1, -1, -1]])
        par.append([[2.0, 0, 0, 0, 0, 0]])
    F = np.zeros((1 if vdp else 2, n))
    F[:, pos[a // 2]] = F[:, pos[a + b // 2]] = 1.0
    return I.FEModel("two_chains", M, D, K, np.concatenate(typ).astype(np.int32), np.concatenate(dof).astype(np.int32),
                     np.concatenate(par).astype(float), F, I._first_mode(M, K))


def _fse():
    from paper_2508_06302_gb300 import fse
    fse.load()
    return fse


@pytest.mark.parametrize("use_graph", [False, True])
def test_batch_of_divided_models(use_graph):
    fse = _fse()
    shell, chains = I.flat_shell(nx=6, ny=4), two_chains(45, 33)
    ctxs = [fse.Context(m, 2, S, H, [I.GOLDEN], 24, newton_tol=0, newton_maxit=6, precision=p)
            for m, S, H, p in ((shell, [5], [2], "fp64"), (shell, [9], [4], "mixed_fp32"), (chains, [6], [2], "fp64"))]
    om = np.array([shell.omega_n1, shell.omega_n1, 1.1 * chains.omega_n1])
    batch = fse.Batch(ctxs, use_graph=use_graph)
    for seed in (1, 2):
        Zs = [I.random_coeffs(c.n, c.U, 1e-4, seed=seed + 10 * k) for k, c in enumerate(ctxs)]
        Rb, st, rc = batch.residual_jacobian(Zs, om, want_jacobian=True)
        assert rc == 0 and np.all(st == 0)
        mono = [c.monodromy() for c in ctxs]
        for k, c in enumerate(ctxs):
            R, _, _, rc = c.residual_jacobian(Zs[k], om[k])
            assert rc == 0 and np.array_equal(R, Rb[k])
            Phi, dz = c.monodromy()
            assert np.array_equal(Phi, mono[k][0]) and np.array_equal(dz, mono[k][1])
    batch.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
def test_shards_of_a_divided_model(precision):
    fse = _fse()
    from paper_2508_06302_gb300.shard import shard_range
    m = two_chains(70, 33)
    w1 = 1.1 * m.omega_n1
    kw = dict(newton_tol=0, newton_maxit=6, precision=precision)
    full = fse.Context(m, 2, [13], [5], [I.GOLDEN], 24, **kw)
    Z, V = I.random_coeffs(m.n, full.U, 1e-3, seed=3), I.random_coeffs(m.n, full.U, 1.0, seed=4)
    want = (full.residual_jacobian(Z, w1)[0], full.jacobian_apply(V)[0], full.jacobian_domega())
    sums = [-Z, -V, 0.0]
    for r in range(3):
        with fse.Context(m, 2, [13], [5], [I.GOLDEN], 24, shard=shard_range(13, r, 3), **kw) as sh:
            sums[0] = sums[0] + sh.residual_jacobian(Z, w1)[0]
            sums[1] = sums[1] + sh.jacobian_apply(V)[0]
            sums[2] = sums[2] + sh.jacobian_domega()
    for a, b in zip(sums, want):
        assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
    full.close()


def test_unknown_frequency_update_of_a_divided_model():
    fse = _fse()
    m = two_chains(40, 33, vdp=True)
    w1, rho = 1.1 * m.omega_n1, [2.3]
    Z = I.random_coeffs(m.n, 5, 1e-3, seed=3)
    Zr, rr, rn, _ = UF.newton_step_unknown(m, [5], [2], 12, rho, Z, w1, [0], tol=0, maxit=10)
    with fse.Context(m, 2, [5], [2], rho, 12, newton_tol=0.0, newton_maxit=10) as ctx:
        ctx.set_linear_solver("dense")
        Zn, rho_n, res, rc = ctx.newton_step_unknown(Z, w1, rho, [0])
    assert abs(res - rn) <= 1e-10 * rn
    assert np.linalg.norm(Zn - Zr) <= 1e-8 * np.linalg.norm(Zr - Z)
    assert abs(rho_n[0] - rr[0]) <= 1e-8 * max(abs(rr[0] - rho[0]), 1e-3)
