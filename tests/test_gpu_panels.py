"""Models whose dofs fall into decoupled components: the tangents are stored and solved panel by
panel, in an internal numbering, while every argument and result keeps the caller's dof order.
Parity with the CPU oracle, which knows nothing of components, over all consumers of the monodromies;
and undivided models at the half-bandwidths where the blocked solves and the panel factor change form
(the shells of the other parity cases divide).  Tolerances as in test_gpu_parity.py: FP64 results 1e-10
relative, FP32 monodromies 1e-3, tensor-core against FP32 FMA solves 1e-4.
"""
import math

import numpy as np
import pytest

from oracle import fse_oracle as O
from oracle import hypertime as HT
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _fse():
    from paper_2508_06302_gb300 import fse
    fse.load()
    return fse


def interleaved(sizes, vdp=False):
    """Independent chains of the given lengths, their dofs dealt out in turn (so that no component is
    contiguous), cubic springs inside each; vdp: a self-excited damper on the second chain."""
    n = sum(sizes)
    dof = [[] for _ in sizes]
    for i, (_, c) in enumerate(sorted(((k + 0.5) / sz, c) for c, sz in enumerate(sizes) for k in range(sz))):
        dof[c].append(i)
    K, M = np.zeros((n, n)), np.zeros((n, n))
    typ, nd, par, F = [], [], [], np.zeros((2, n))
    for c, d in enumerate(dof):
        k = 1e4 * (1 + 0.3 * c)
        for a, x in enumerate(d):
            K[x, x] = 2 * k
            M[x, x] = 1.0 + 0.1 * c
            if a:
                K[x, d[a - 1]] = K[d[a - 1], x] = -k
                typ.append(I.NL_CUBIC_DIFF)
                nd.append([d[a - 1], x, -1, -1, -1, -1])
                par.append([5e7, 0, 0, 0, 0, 0])
        typ.append(I.NL_CUBIC_GROUND)
        nd.append([d[0], -1, -1, -1, -1, -1])
        par.append([1e8, 0, 0, 0, 0, 0])
        F[0, d[len(d) // 2]], F[1, d[len(d) // 2]] = 1.0, 0.5
    if vdp:
        typ.append(I.NL_VDP)
        nd.append([dof[1][0], -1, -1, -1, -1, -1])
        par.append([2.0, 0, 0, 0, 0, 0])
    return I.FEModel("interleaved", M, 0.5 * M + 5e-5 * K, K, np.array(typ, np.int32), np.array(nd, np.int32),
                     np.array(par, float), F, I._first_mode(M, K))


MODELS = {
    # panels of 1 to 4; the last one shared by several small components; blocks of 32 rows filled up,
    # exactly full and one over
    "two": lambda: interleaved([64, 33]),
    "shared": lambda: interleaved([40, 32, 31, 5, 2, 1, 1]),
    "vdp": lambda: interleaved([45, 33, 8], vdp=True),
    "singles": lambda: interleaved([1] * 70),
}


def _case(mk, precision, S1=12):
    m = mk()
    w1 = 1.1 * m.omega_n1
    rho = [I.GOLDEN]
    ctx = _fse().Context(m, 2, [5], [2], rho, S1, newton_tol=0.0, newton_maxit=12, precision=precision)
    Z = I.random_coeffs(m.n, 5, 1e-3, seed=3)
    return m, w1, O.FSEProblem(m, [5], [2], S1, rho), ctx, Z


def _close(a, b, tol):
    a, b = np.asarray(a), np.asarray(b)
    assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("name", list(MODELS))
def test_panels_fp64(name):
    m, w1, prob, ctx, Z = _case(MODELS[name], "fp64")
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=True, dense=True, tol=0, maxit=12)
    R, st, it, rc = ctx.residual_jacobian(Z, w1)
    assert rc == 0
    _close(R, ref.R, 1e-10)
    Phi, dz = ctx.monodromy()
    _close(Phi, ref.Phi, 1e-10)
    _close(dz, ref.dz_dw, 1e-10)
    P1, d1 = ctx.monodromy_traj(3)
    assert np.array_equal(P1, Phi[3]) and np.array_equal(d1, dz[3])
    V = np.random.default_rng(1).standard_normal((2, Z.size))
    _close(ctx.jacobian_apply(V), V @ ref.J.T, 1e-10)
    _close(ctx.jacobian_domega(), ref.dR_dw, 1e-10)
    _close(ctx.jacobian_dense(), ref.J, 1e-10)
    # residual-only evaluations keep older factors; to the fixed 12 Newton iterations they agree
    _close(ctx.residual_jacobian(Z, w1, want_jacobian=False)[0], ref.R, 1e-10)
    dZ = np.linalg.solve(ref.J, -ref.R)
    ctx.set_linear_solver("dense")
    Zn, rn, rc = ctx.newton_step(Z, w1)
    _close(Zn - Z, dZ, 1e-8)
    h = min(4, 2 * m.n)
    ref_s = O.lyapunov(prob, ref.Phi, w1, N_Ly=3, h=h)
    np.testing.assert_allclose(ctx.lyapunov(Z, w1, 3, h), ref_s, rtol=1e-8, atol=1e-6)
    ctx.close()


@pytest.mark.parametrize("name", list(MODELS))
def test_panels_fp32_and_tensor_core(name):
    m, w1, prob, ctx, Z = _case(MODELS[name], "mixed_fp32")
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=True, dense=False, tol=0, maxit=12)
    out = {}
    for kind in ("tc", "simt"):
        ctx.set_tangent_solve(kind)
        R, st, it, rc = ctx.residual_jacobian(Z, w1)
        assert rc == 0
        _close(R, ref.R, 1e-10)
        out[kind] = ctx.monodromy()[0]
        _close(out[kind], ref.Phi, 1e-3)
    _close(out["tc"], out["simt"], 1e-4)
    ctx.close()


def test_panels_hypertime():
    m, w1, prob, ctx, Z = _case(MODELS["shared"], "fp64")
    rng = np.random.default_rng(5)
    z0 = 1e-3 * rng.standard_normal((5, 2 * m.n))
    RT, J = HT.residual_jacobian_hypertime(prob, z0, w1, want_jacobian=True, tol=0, maxit=12)
    _close(ctx.residual_jacobian_hypertime(z0, w1)[0], RT, 1e-10)
    V = rng.standard_normal(z0.shape)
    _close(ctx.jacobian_apply_hypertime(V).reshape(-1), J @ V.reshape(-1), 1e-10)
    ctx.close()


# plates couple all their dofs: half-bandwidth 3 (ny - 1) + 5
@pytest.mark.parametrize("ny,precision", [(5, "fp64"), (16, "fp64"), (30, "mixed_fp32"), (31, "mixed_fp32"),
                                          (32, "mixed_fp32")])
def test_undivided_band_limits(ny, precision):
    m = I.kirchhoff_plate(nx=3, ny=ny, n_springs=3, e_count=2)
    w1 = 1.1 * m.omega_n1
    prob = O.FSEProblem(m, [5], [2], 12, [I.GOLDEN])
    Z = I.random_coeffs(m.n, 5, 1e-4, seed=7)
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=True, dense=False, tol=0, maxit=12)
    ctx = _fse().Context(m, 2, [5], [2], [I.GOLDEN], 12, newton_tol=0.0, newton_maxit=12, precision=precision)
    kinds = ["simt"] + (["tc"] if precision != "fp64" and ctx.band <= 96 else [])
    for kind in kinds:
        ctx.set_tangent_solve(kind)
        R, st, it, rc = ctx.residual_jacobian(Z, w1)
        assert rc == 0
        _close(R, ref.R, 1e-10)
        _close(ctx.monodromy()[0], ref.Phi, 1e-10 if precision == "fp64" else 1e-3)
    ctx.close()


def test_limits_stay_the_callers_numbering():
    """The size limits are those of the caller's numbering, whatever the components would allow."""
    fse = _fse()
    m = I.flat_shell(nx=3, ny=18)
    with fse.Context(m, 2, [5], [2], [I.GOLDEN], 20, precision="mixed_fp32") as ctx:
        assert ctx.band == 110
        with pytest.raises(fse.FSEError) as ei:
            ctx.set_tangent_solve("tc")
        assert ei.value.code == fse.FSE_EINVAL
    with pytest.raises(fse.FSEError) as ei:
        fse.Context(m, 2, [5], [2], [I.GOLDEN], 20, precision="fp64")
    assert ei.value.code == fse.FSE_EINVAL
