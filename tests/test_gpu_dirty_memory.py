"""Contexts created on memory that earlier programs filled: nothing the kernels read may be left over.
Models with wide panels whose sizes are no multiples of 32 rows (inert rows between the panels), in both
precisions; against the oracle with the tolerances of test_gpu_parity.py, and
equal bit for bit whatever the memory held."""
import ctypes

import numpy as np
import pytest

from oracle import fse_oracle as O
from paper_2508_06302_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def fill_device(word):
    """Fill device memory with a 32-bit word, in blocks of the sizes a context asks for, and give three of
    four blocks back; the fourth ones, returned, keep the driver from clearing what lies between."""
    import torch
    torch.zeros(1, device="cuda")   # the CUDA context the library uses
    cuda = ctypes.CDLL("libcuda.so.1")
    kept = []
    for size, count in ((1 << 12, 800), (1 << 15, 400), (1 << 17, 200), (1 << 18, 120), (600000, 80)):
        ptrs = []
        for _ in range(count):
            p = ctypes.c_uint64()
            assert cuda.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(size)) == 0
            ptrs.append(p)
            assert cuda.cuMemsetD32_v2(p, ctypes.c_uint32(word), ctypes.c_size_t(size // 4)) == 0
        torch.cuda.synchronize()
        for k, p in enumerate(ptrs):
            if k % 4:
                assert cuda.cuMemFree_v2(p) == 0
            else:
                kept.append(p)
    return lambda: [cuda.cuMemFree_v2(p) for p in kept]


# zeros; FP64 and FP32 values around 1e29 and 1e4; NaN in both
WORDS = (0, 0x46000000, 0xffffffff)


@pytest.mark.parametrize("nx,ny,precision", [(6, 4, "fp64"), (8, 7, "fp64"), (4, 14, "fp64"), (8, 7, "mixed_fp32"),
                                             (3, 17, "mixed_fp32")])
def test_context_on_used_memory(nx, ny, precision):
    from paper_2508_06302_gb300 import fse
    m = I.flat_shell(nx=nx, ny=ny)
    w1 = m.omega_n1
    prob = O.FSEProblem(m, [5], [2], 40, [I.GOLDEN])
    Z = I.random_coeffs(m.n, 5, 1e-5, seed=5)
    ref = O.residual_jacobian(prob, Z, w1, want_jacobian=True, dense=False, tol=0, maxit=8, n_steps=4)
    first = None
    for word in WORDS:
        release = fill_device(word)
        with fse.Context(m, 2, [5], [2], [I.GOLDEN], 40, newton_tol=0.0, newton_maxit=8, precision=precision) as ctx:
            ctx.set_steps(4)
            R, st, it, rc = ctx.residual_jacobian(Z, w1)
            assert rc == 0, hex(word)
            Phi, dz = ctx.monodromy()
            Rr, st, it, rc = ctx.residual_jacobian(Z, w1, want_jacobian=False)
            assert rc == 0, hex(word)
        release()
        out = (R, Phi, dz, Rr)
        assert np.linalg.norm(R - ref.R) <= 1e-10 * np.linalg.norm(ref.R)
        assert np.linalg.norm(Rr - ref.R) <= 1e-10 * np.linalg.norm(ref.R)
        tol = 1e-10 if precision == "fp64" else 1e-3
        assert np.linalg.norm(Phi - ref.Phi) <= tol * np.linalg.norm(ref.Phi)
        first = out if first is None else first
        assert all(np.array_equal(a, b) for a, b in zip(out, first)), hex(word)


def test_newton_updates_ignore_what_their_buffers_held():
    """Right-hand sides are formed as -R in buffers that hold anything: fresh memory full of NaN (unknown
    frequency, hyper-time), or the NaN product of an earlier call (dense and GMRES updates)."""
    from paper_2508_06302_gb300 import fse
    v, m = I.van_der_pol(omega_n=10.0, eps=0.2, F=(10.0,)), I.chain(6)
    wv, wm = 10.0 / 2.7, 1.1 * m.omega_n1
    Zv, Zm = I.random_coeffs(v.n, 7, 0.3, seed=3), I.random_coeffs(m.n, 5, 1e-3, seed=3)
    z = np.random.default_rng(1).standard_normal((5, 2 * m.n)) * 1e-3
    out = []
    for word in WORDS:
        release = fill_device(word)
        with fse.Context(v, 2, [8], [3], [2.7], 24, newton_tol=0.0, newton_maxit=8) as ctx:
            Z, rho, rn, rc = ctx.newton_step_unknown(Zv, wv, [2.7], [0])
        with fse.Context(m, 2, [5], [2], [I.GOLDEN], 24, newton_tol=0.0, newton_maxit=8) as ctx:
            zn = ctx.newton_step_hypertime(z, wm)[0]
            ctx.jacobian_apply_hypertime(np.full((1,) + z.shape, np.nan))
            zh = ctx.newton_step_hypertime(z, wm)[0]
            ctx.residual_jacobian(Zm, wm)
            Zd = []
            for solver in ("dense", "gmres"):
                ctx.set_linear_solver(solver)
                ctx.jacobian_apply(np.full((2, Zm.size), np.nan))
                Zd.append(ctx.newton_step(Zm, wm)[0])
        release()
        out.append((Z, rho, zn, zh, *Zd))
        assert all(np.all(np.isfinite(a)) for a in out[-1]), hex(word)
        assert np.array_equal(zn, zh)
        assert all(np.array_equal(a, b) for a, b in zip(out[-1], out[0])), hex(word)
