"""Performance cases: the calls a user of the framework makes on the way to a quasi-periodic torus.

A case names a structural model and its mesh, the trajectory grid of the torus, the Newmark steps and
the call that is timed:

  jacobian   one residual + Jacobian evaluation (Eq. 16, 22) and the products the outer solve takes
             from it (J v for two vectors; dR/dw_1 where the tangents are FP64: the FP32 column is
             too coarse to be compared)
  residual   one residual-only evaluation (what the chord corrector of a continuation repeats)
  products   J v on the stored monodromies (what every GMRES iteration of the outer solve repeats)
  newton     one whole Newton update of Z(0): evaluation, Jacobian, outer solve
  lyapunov   the Lyapunov exponents of a torus (App. F): evaluation and propagation
  hypertime  residual + Jacobian of the hyper-time form (Sec. 3.4) and its J_T v

The large models are integrated over the first `run_steps` Newmark steps of the period (fse_set_steps,
the entry point for sampled timing): a period repeats the same step `steps` times.

A mixed-precision context keeps its tangents in FP32, so what is read from them is handed on in that
type; the residual is FP64 in every mode.
"""
import math

import numpy as np
import torch

from paper_2508_06302_gb300 import fse, inputs

RHO = {2: [inputs.GOLDEN], 3: [math.sqrt(2.0), math.sqrt(3.0)]}


def listed():
    return [
        # the smallest whole call: one Newton update of the 18-dof beam torus with the dense outer
        # solve, the default for problems of this size; launches and latency are what a user waits for
        dict(name="beam18_newton", call="newton", model="beam", m1=10, m2=0, s2=16, h2=7, s3=0, h3=0, steps=128,
             run_steps=0, precision="fp64", solver="dense", w=1.1),
        # the same torus in mixed precision, over a quarter of its period, as a corrector of a sweep calls it
        dict(name="beam18_jacobian_mixed", call="jacobian", model="beam", m1=10, m2=0, s2=16, h2=7, s3=0, h3=0,
             steps=128, run_steps=32, precision="mixed_fp32", w=1.1),
        # stability of a torus of a small shell: exponents in FP64, the certified form
        dict(name="shell90_lyapunov", call="lyapunov", model="shell", m1=6, m2=4, s2=15, h2=7, s3=0, h3=0, steps=60,
             run_steps=0, precision="fp64", n_ly=100, h=32, w=1.0),
        # the nearly undamped von Karman beam, which needs FP64 tangents
        dict(name="vkbeam447_jacobian", call="jacobian", model="vkbeam", m1=150, m2=0, s2=64, h2=31, s3=0, h3=0,
             steps=512, run_steps=48, precision="fp64", w=1.1),
        # d = 3: many trajectories of a mid-size plate, mixed precision
        dict(name="plate243_jacobian_mixed", call="jacobian", model="plate", m1=10, m2=10, s2=16, h2=7, s3=16, h3=7,
             steps=400, run_steps=16, precision="mixed_fp32", w=1.1),
        # the same plate, residual only, in plain FP64 (state path alone)
        dict(name="plate243_residual", call="residual", model="plate", m1=10, m2=10, s2=16, h2=7, s3=16, h3=7,
             steps=400, run_steps=40, precision="fp64", w=1.1),
        # the 1872-dof shell of the benchmark, residual + Jacobian: the largest call
        dict(name="shell1872_jacobian_mixed", call="jacobian", model="shell", m1=25, m2=14, s2=64, h2=31, s3=0, h3=0,
             steps=1000, run_steps=24, precision="mixed_fp32", w=1.0),
        # its residual-only evaluation (2 to 4 of them per continuation point)
        dict(name="shell1872_residual_mixed", call="residual", model="shell", m1=25, m2=14, s2=64, h2=31, s3=0,
             h3=0, steps=1000, run_steps=48, precision="mixed_fp32", w=1.0),
        # the products of its GMRES solve (about 200 per continuation point)
        dict(name="shell1872_products_mixed", call="products", model="shell", m1=25, m2=14, s2=64, h2=31, s3=0,
             h3=0, steps=1000, run_steps=4, precision="mixed_fp32", nvec=8, w=1.0),
        # a mid-size shell at ragged sizes (37 trajectories, 61 steps), a whole FP64 Newton update with GMRES
        dict(name="shell360_newton_gmres", call="newton", model="shell", m1=11, m2=7, s2=37, h2=18, s3=0, h3=0,
             steps=61, run_steps=0, precision="fp64", solver="gmres", w=0.9),
        # a mesh numbered across its long side: half-bandwidth 98, beyond the narrow solves
        dict(name="shell540_wideband_mixed", call="jacobian", model="shell", m1=7, m2=16, s2=21, h2=9, s3=0, h3=0,
             steps=300, run_steps=24, precision="mixed_fp32", w=0.95),
        # the hyper-time form on a small plate with more samples than coefficients, FP64
        dict(name="plate72_hypertime", call="hypertime", model="plate", m1=7, m2=5, s2=19, h2=7, s3=0, h3=0, steps=90,
             run_steps=0, precision="fp64", w=1.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["jacobian", "jacobian", "jacobian", "residual", "residual", "products", "newton", "lyapunov",
                       "hypertime"])
    full = call in ("newton", "lyapunov", "hypertime")     # whole periods: smaller models
    model = rng.choice(["beam", "vkbeam", "plate", "shell", "shell"])
    if full and model == "vkbeam":
        model = "beam"                                      # its tori are far from a first Newton update
    if call == "lyapunov":
        model = "shell"                                     # a beam's trailing exponents need more than 64 bits
    precision = rng.choice(["fp64", "mixed_fp32"])
    if model == "vkbeam" or full:
        precision = "fp64"
    m2 = 0
    if model == "beam":
        m1 = _log(rng, 3, 40)
    elif model == "vkbeam":
        m1 = 2 * _log(rng, 5, 75)
    elif model == "plate":
        m1, m2 = rng.randint(3, 7 if full else 12), rng.randint(3, 7 if full else 12)
    else:
        m2 = rng.randint(4 if call == "lyapunov" else 3, 6 if full else (9 if precision == "fp64" else 16))
        m1 = rng.randint(3, 7) if full or m2 > 14 else _log(rng, max(3, m2 // 2), 25)
    case = dict(call=call, model=model, m1=m1, m2=m2, s3=0, h3=0, precision=precision,
                w=round(rng.uniform(0.85, 1.15), 3))
    n = _dofs(case)
    if model == "plate" and not full and rng.random() < 0.5:
        h2, h3 = rng.randint(1, 6), rng.randint(1, 6)
        case.update(h2=h2, s2=2 * h2 + 1 + rng.randint(0, 1), h3=h3, s3=2 * h3 + 1 + rng.randint(0, 1))
    else:
        h2 = _log(rng, 3 if call == "lyapunov" else 1, 9 if full else 31)
        case.update(h2=h2, s2=2 * h2 + 1 + rng.randint(0, 2))
    N = case["s2"] * max(1, case["s3"])
    # FP32 tangents lose about steps / 1000 x 1e-6 per step taken: past 360 they say little after a few steps
    case["steps"] = rng.randint(24, 110) if full else rng.randint(100, 1000 if precision == "fp64" else 360)
    # the tangents of one step cost about N n^2: never more than the largest listed case in all
    most = 24 * 64 * 1872 * 1872 / (30 if precision == "fp64" else 2)
    case["run_steps"] = 0 if full else max(4, min(rng.randint(8, 40 if precision == "fp64" else 16), int(most / (N * n * n))))
    if call == "products":
        case.update(run_steps=4, nvec=rng.randint(1, 12))
    if call == "newton":
        case["solver"] = "dense" if 2 * n * (2 * h2 + 1) <= 1200 else "gmres"
    if call == "lyapunov":
        case.update(n_ly=_log(rng, 20, 200), h=rng.randint(2, min(32, 2 * n)))
    return case


def _dofs(case):
    m1, m2 = case["m1"], case["m2"]
    return {"beam": 2 * (m1 - 1), "vkbeam": 3 * (m1 - 1), "plate": 3 * (m1 - 1) * (m2 - 1),
            "shell": 6 * (m1 - 1) * (m2 - 1)}[case["model"]]


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------

_models = {}      # meshes by size: assembled once per process, as a program does with its own mesh
_responses = {}


def _mesh(case):
    key = (case["model"], case["m1"], case["m2"], bool(case["s3"]))
    if key not in _models:
        m1, m2 = case["m1"], case["m2"]
        if case["model"] == "beam":
            m = inputs.eb_beam(n_el=m1)
        elif case["model"] == "vkbeam":
            m = inputs.vk_beam(n_el=m1, F1=0.05, F2=0.05)
        elif case["model"] == "plate":
            nodes = (m1 - 1) * (m2 - 1)
            m = inputs.kirchhoff_plate(nx=m1, ny=m2, n_springs=max(1, nodes // 2), e_count=3 if case["s3"] else 2)
        else:
            m = inputs.flat_shell(nx=m1, ny=m2)
        _models[key] = m
    return key, _models[key]


def _harmonics(case):
    """Harmonic table of App. B (Eq. B1-B2), the zero row left out."""
    rows = [[k] for k in range(1, case["h2"] + 1)] + [[0]]
    if case["s3"]:
        nxt = [r + [-k] for k in range(1, case["h3"] + 1) for r in rows[:-1]]
        for k in list(range(1, case["h3"] + 1)) + [0]:
            nxt += [r + [k] for r in rows]
        rows = nxt
    return np.array(rows[:-1], dtype=np.int64).reshape(len(rows) - 1, 2 if case["s3"] else 1)


def _response(case, omega):
    """Linear steady responses (displacement, derivative w.r.t. phi_1) of the forcing components."""
    key, m = _mesh(case)
    key = key + (omega,)
    if key not in _responses:
        out = []
        for F, r in zip(m.F, [1.0] + RHO[3 if case["s3"] else 2]):
            q = np.linalg.solve(m.K + 1j * (r * omega) * m.D - (r * omega) ** 2 * m.M, F)
            out.append((q, 1j * r * q))
        _responses[key] = out
    return _responses[key]


def _torus(case, omega, rng):
    """Fourier coefficients of a smooth torus near the linear response: seeded amplitudes and phases,
    higher harmonics falling off by ten per order (state-major, as Eq. 11)."""
    resp = _response(case, omega)
    ktab = _harmonics(case)
    n = _dofs(case)
    C = np.zeros((2 * n, 2 * len(ktab) + 1))

    def seeded():
        return rng.uniform(0.6, 1.4) * np.exp(2j * math.pi * rng.uniform(-0.2, 0.2))

    c = seeded()
    C[:n, 0], C[n:, 0] = (c * resp[0][0]).real, (c * resp[0][1]).real
    for l, k in enumerate(ktab):
        order = int(np.abs(k).sum())
        j = 1 + int(np.argmax(np.abs(k)))
        if order == 1 and j < len(resp):
            c, (q, u) = seeded(), resp[j]
        else:
            c = 10.0 ** -min(order, 6) * (rng.standard_normal() + 1j * rng.standard_normal())
            q, u = resp[rng.integers(len(resp))]
        C[:n, 1 + 2 * l], C[:n, 2 + 2 * l] = (c * q).real, -(c * q).imag
        C[n:, 1 + 2 * l], C[n:, 2 + 2 * l] = (c * u).real, -(c * u).imag
    return C


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    _, mesh = _mesh(case)
    p = mesh.nl_p.copy()
    if case["model"] != "vkbeam":                 # seeded spring stiffnesses
        p[:, 0] *= rng.uniform(0.8, 1.25, p.shape[0])
    model = inputs.FEModel(mesh.name, mesh.M, mesh.D, mesh.K, mesh.nl_type, mesh.nl_dof, p, mesh.F, mesh.omega_n1)
    omega = case["w"] * model.omega_n1
    C = _torus(case, omega, rng)
    x = dict(model=model, omega=omega, Z=C.reshape(-1))
    nv = case.get("nvec", 2)
    if case["call"] == "hypertime":
        x["z"] = (_grid(case)[1] @ C.T).copy()    # start points of the trajectories
        x["V"] = rng.standard_normal((nv,) + x["z"].shape)
    elif case["call"] in ("jacobian", "products"):
        x["V"] = rng.standard_normal((nv, x["Z"].size))
    return x


def _grid(case):
    """Sample phases (Eq. D1, phi_2 fastest) and Gamma (Eq. D2)."""
    S = [case["s2"]] + ([case["s3"]] if case["s3"] else [])
    N = int(np.prod(S))
    s = np.arange(N)
    ph = np.stack([2 * math.pi * (s % S[0]) / S[0]] + ([2 * math.pi * (s // S[0]) / S[1]] if len(S) > 1 else []), 1)
    arg = ph @ _harmonics(case).T
    G = np.ones((N, 2 * arg.shape[1] + 1))
    G[:, 1::2], G[:, 2::2] = np.cos(arg), np.sin(arg)
    return ph, G


def prepare(case, seed):
    x = _inputs(case, seed)
    d = 3 if case["s3"] else 2
    ctx = fse.Context(x["model"], d, [case["s2"]] + ([case["s3"]] if d == 3 else []),
                      [case["h2"]] + ([case["h3"]] if d == 3 else []), RHO[d], case["steps"],
                      precision=case["precision"])
    ctx.set_steps(case["run_steps"])
    if case["call"] == "newton":
        ctx.set_linear_solver(case["solver"], rel_tol=1e-12)
    if case["call"] == "products":
        ctx.residual_jacobian(x["Z"], x["omega"], want_jacobian=True)
    x.update(ctx=ctx, call=case["call"], case=case, mixed=case["precision"] != "fp64")
    return x


def run(x):
    ctx, call = x["ctx"], x["call"]
    own = (lambda a: a.astype(np.float32)) if x["mixed"] else (lambda a: a)
    if call == "jacobian":
        R = ctx.residual_jacobian(x["Z"], x["omega"], want_jacobian=True)[0]
        out = {"R": R, "Jv": own(ctx.jacobian_apply(x["V"]))}
        if not x["mixed"]:
            out["dRdw"] = ctx.jacobian_domega()
        return out
    if call == "residual":
        return {"R": ctx.residual_jacobian(x["Z"], x["omega"], want_jacobian=False)[0]}
    if call == "products":
        return {"Jv": own(ctx.jacobian_apply(x["V"]))}
    if call == "newton":
        Z, rn, _ = ctx.newton_step(x["Z"], x["omega"])
        return {"Z": own(Z), "res": float(rn)}
    if call == "lyapunov":
        return {"sigma": ctx.lyapunov(x["Z"], x["omega"], x["case"]["n_ly"], x["case"]["h"])}
    RT = ctx.residual_jacobian_hypertime(x["z"], x["omega"], want_jacobian=True)[0]
    return {"RT": RT, "Jv": own(ctx.jacobian_apply_hypertime(x["V"]))}


def work(case):
    """Bytes: the model, the call's vectors and, with a Jacobian, the monodromies once; where the
    tangents of all trajectories exceed what stays on the chip (about 100 MB), they are read and
    written once per Newmark step.  Flops: banded factor, solves and sparse products of the state
    (two Newton iterations) and of the tangents; the outer solve."""
    _, m = _mesh(case)
    n = m.n
    pat = (m.M != 0) | (m.D != 0) | (m.K != 0)
    ij = np.nonzero(pat)
    b = max(int(np.abs(ij[0] - ij[1]).max()), 1)
    nnz = len(ij[0])
    N, U = case["s2"] * max(1, case["s3"]), 2 * len(_harmonics(case)) + 1
    steps = case["run_steps"] or case["steps"]
    T = 8 if case["precision"] == "fp64" else 4
    call = case["call"]
    P = 2 * n + 1
    phi = N * 2 * n * P * T
    vec = 8 * 2 * n * (N if call == "hypertime" else U)
    nv = case.get("nvec", 2)
    state = steps * N * (n * b * b + 3 * 4 * n * b + 10 * nnz)
    aft = 4 * N * U * n * 2
    prod = nv * (2 * N * 4 * n * n + 2 * aft)
    byts, flops = 3 * 8 * nnz + 2 * vec, aft * 2
    if call == "products":
        return {"bytes": phi + 2 * nv * vec, "flops": prod}
    flops += state
    if call != "residual":
        flops += steps * N * P * (4 * nnz + 4 * n * b)
        byts += 2 * phi * steps if phi > 1e8 else phi
    if call in ("jacobian", "hypertime"):
        byts += 2 * nv * vec
        flops += prod
    if call == "newton":
        flops += (2 * n * U) ** 3 * 2 / 3 if case["solver"] == "dense" else 30 * (8 * N * n * n + 2 * aft)
    if call == "lyapunov":
        flops += case["n_ly"] * (2 * N * 4 * n * n * case["h"] + 4 * 2 * n * case["h"] ** 2)
    return {"bytes": byts, "flops": flops}


# ----------------------------------------------------------------------------------------------
# the same results in 64 bits: Newmark with the acceleration kept (Eq. E5-E7 and their derivatives),
# full Newton, block-tridiagonal Cholesky over all trajectories at once
# ----------------------------------------------------------------------------------------------

class _Elements:
    """f_nl and its tangent, all trajectories at once."""

    def __init__(self, m, dev):
        self.n, self.parts = m.n, []
        for t in (1, 2, 3):
            e = np.nonzero(m.nl_type == t)[0]
            nd = {1: 1, 2: 2, 3: 6}[t]
            if len(e):
                self.parts.append((t, torch.tensor(np.where(m.nl_dof[e, :nd] < 0, m.n, m.nl_dof[e, :nd]), device=dev),
                                   torch.tensor(m.nl_p[e], device=dev)))
        xg, wg = np.polynomial.legendre.leggauss(5)
        self.xg, self.wg = [float(v) for v in xg], [float(v) for v in wg]

    def both(self, q, tangent=True):
        """(f (N, n), [(dofs, k (N, el, nd, nd))])"""
        N, n = q.shape
        qp = torch.cat([q, q.new_zeros(N, 1)], 1)
        f = q.new_zeros(N, n + 1)
        ks = []
        for t, dof, p in self.parts:
            x = qp[:, dof]
            if t == 1:
                fe = p[:, :1] * x ** 3
                ke = (3 * p[:, :1] * x ** 2)[..., None]
            elif t == 2:
                s = x[..., :1] - x[..., 1:]
                sg = x.new_tensor([1.0, -1.0])
                fe = p[:, :1] * s ** 3 * sg
                ke = (3 * p[:, :1] * s ** 2)[..., None] * sg[:, None] * sg[None, :]
            else:
                EA, L = p[:, 0], p[:, 1]
                fe = x.new_zeros(x.shape)
                ke = x.new_zeros(x.shape + (6,))
                bu = x.new_zeros(len(L), 6)
                bu[:, 0], bu[:, 3] = -1 / L, 1 / L
                du = (x * bu).sum(-1)
                for xi, wt in zip(self.xg, self.wg):
                    s = 0.5 * (xi + 1)
                    bw = x.new_zeros(len(L), 6)
                    bw[:, 1], bw[:, 2] = (-6 * s + 6 * s * s) / L, 1 - 4 * s + 3 * s * s
                    bw[:, 4], bw[:, 5] = (6 * s - 6 * s * s) / L, -2 * s + 3 * s * s
                    c = 0.5 * L * wt * EA
                    wp = (x * bw).sum(-1)
                    fe += (c * 0.5 * wp ** 2)[..., None] * bu + (c * (du * wp + 0.5 * wp ** 3))[..., None] * bw
                    ke += (c * wp)[..., None, None] * (bu[:, :, None] * bw[:, None, :] + bw[:, :, None] * bu[:, None, :])
                    ke += (c * (du + 1.5 * wp ** 2))[..., None, None] * (bw[:, :, None] * bw[:, None, :])
            f.index_add_(1, dof.reshape(-1), fe.reshape(N, -1))
            ks.append((dof, ke))
        return f[:, :n], ks if tangent else None


class _Blocks:
    """Cholesky factor of S + K_t as a block-tridiagonal matrix, batched over the trajectories."""

    def __init__(self, S, ks, N, b):
        n = S.shape[0]
        s = max(b, 12)
        nb = -(-n // s)
        A = S.new_zeros(N, nb * s + 1, nb * s + 1)
        A[:, :n, :n] = S
        for dof, ke in ks:
            d = torch.where(dof < n, dof, torch.full_like(dof, nb * s))
            rows = d[:, :, None].expand(ke.shape[1:]).reshape(-1)
            cols = d[:, None, :].expand(ke.shape[1:]).reshape(-1)
            A.view(N, -1).index_add_(1, rows * (nb * s + 1) + cols, ke.reshape(N, -1))
        i = torch.arange(n, nb * s, device=S.device)
        A[:, i, i] = 1.0
        self.n, self.s, self.nb, self.C, self.G = n, s, nb, [], []
        D = A[:, :s, :s].contiguous()
        for k in range(nb):
            self.C.append(torch.linalg.cholesky(D))
            if k + 1 < nb:
                a = A[:, (k + 1) * s:(k + 2) * s, k * s:(k + 1) * s]
                g = torch.linalg.solve_triangular(self.C[k], a.transpose(1, 2), upper=False).transpose(1, 2).contiguous()
                self.G.append(g)
                D = A[:, (k + 1) * s:(k + 2) * s, (k + 1) * s:(k + 2) * s] - g @ g.transpose(1, 2)

    def solve(self, r):
        s, nb = self.s, self.nb
        y = torch.cat([r, r.new_zeros(r.shape[0], nb * s - self.n, r.shape[2])], 1)
        for k in range(nb):
            v = y[:, k * s:(k + 1) * s]
            if k:
                v = v - self.G[k - 1] @ y[:, (k - 1) * s:k * s]
            y[:, k * s:(k + 1) * s] = torch.linalg.solve_triangular(self.C[k], v, upper=False)
        for k in reversed(range(nb)):
            v = y[:, k * s:(k + 1) * s]
            if k + 1 < nb:
                v = v - self.G[k].transpose(1, 2) @ y[:, (k + 1) * s:(k + 2) * s]
            y[:, k * s:(k + 1) * s] = torch.linalg.solve_triangular(self.C[k].transpose(1, 2), v, upper=True)
        return y[:, :self.n]


def _integrate(case, m, w, zb, Y, dev):
    """End points of the trajectories from zb (N, 2n), and the tangents of the start directions
    Y (N, 2n, k) with the w_1 derivative as one more column."""
    t64 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    n, N = m.n, zb.shape[0]
    M, D, K, F = t64(m.M), t64(m.D), t64(m.K), t64(m.F)
    ph = t64(_grid(case)[0])
    rho = RHO[3 if case["s3"] else 2]
    h = 2 * math.pi / case["steps"]
    a0, a1, a2 = 4 / h ** 2, 4 / h, 2 / h
    S = w * w * a0 * M + w * a2 * D + K
    ij = torch.nonzero(S)
    b = int((ij[:, 0] - ij[:, 1]).abs().max())
    el = _Elements(m, dev)
    for _, dof, _p in el.parts:
        ok = dof < n
        b = max(b, int((torch.where(ok, dof, dof.amin(1, keepdim=True)).amax(1) - dof.amin(1)).max()))

    def force(phi):
        e = F[0] * math.cos(phi) + torch.zeros(N, n, device=dev, dtype=torch.float64)
        for j in range(1, F.shape[0]):
            e = e + torch.cos(ph[:, j - 1] + rho[j - 1] * phi)[:, None] * F[j]
        return e

    def kt(ks, X):
        out = X.new_zeros(N, n + 1, X.shape[2])
        Xp = torch.cat([X, X.new_zeros(N, 1, X.shape[2])], 1)
        for dof, ke in ks:
            v = torch.einsum("seab,sebk->seak", ke, Xp[:, dof])
            out.index_add_(1, dof.reshape(-1), v.reshape(N, -1, X.shape[2]))
        return out[:, :n]

    q, u = zb[:, :n].clone(), zb[:, n:].clone()
    f, ks = el.both(q)
    LM = torch.linalg.cholesky(w * w * M)
    a = torch.cholesky_solve((force(0.0) - w * u @ D - q @ K - f).T, LM).T
    X = V = W = None
    if Y is not None:
        X, V = (torch.cat([p, p.new_zeros(N, n, 1)], 2) for p in (Y[:, :n], Y[:, n:]))
        r = -(w * (D @ V) + K @ X + kt(ks, X))
        r[:, :, -1] -= 2 * w * a @ M + u @ D
        k = r.shape[2]
        W = torch.cholesky_solve(r.permute(1, 0, 2).reshape(n, -1), LM).reshape(n, N, k).permute(1, 0, 2)
    for step in range(case["run_steps"] or case["steps"]):
        rhs = force((step + 1) * h) + w * w * (a0 * q + a1 * u + a) @ M + w * (a2 * q + u) @ D
        qn = q.clone()
        for _ in range(12):
            f, ks = el.both(qn)
            dq = _Blocks(S, ks, N, b).solve((rhs - qn @ S - f)[:, :, None])[:, :, 0]
            qn = qn + dq
            if float(dq.abs().max()) <= 3e-15 * float(qn.abs().max()):
                break
            if float(dq.abs().max()) <= 1e-9 * float(qn.abs().max()):   # quadratic: one more is exact
                f, ks = el.both(qn)
                qn = qn + _Blocks(S, ks, N, b).solve((rhs - qn @ S - f)[:, :, None])[:, :, 0]
                break
        un, an = a2 * (qn - q) - u, a0 * (qn - q) - a1 * u - a
        if X is not None:
            _, ks = el.both(qn)
            r = w * w * (M @ (a0 * X + a1 * V + W)) + w * (D @ (a2 * X + V))
            r[:, :, -1] -= 2 * w * an @ M + un @ D
            Xn = _Blocks(S, ks, N, b).solve(r)
            V, W = a2 * (Xn - X) - V, a0 * (Xn - X) - a1 * V - W
            X = Xn
        q, u, a = qn, un, an
    end = torch.cat([q, u], 1)
    return end, None if X is None else torch.cat([X, V], 1)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x = _inputs(case, seed)
    m, w, call = x["model"], x["omega"], case["call"]
    n = m.n
    steps = case["run_steps"] or case["steps"]
    G = torch.tensor(_grid(case)[1], device=dev)
    N, U = G.shape
    whole = call in ("newton", "lyapunov")
    if N * n * n * steps * (n / 500 if whole else 1) > 2e10:
        return None
    Gi = 2 * G.T / N
    Gi[0] /= 2
    th = 2 * math.pi * _harmonics(case) @ np.array(RHO[3 if case["s3"] else 2])
    c, s = (torch.tensor(v, device=dev)[:, None] for v in (np.cos(th), np.sin(th)))
    RG = Gi.clone()
    RG[1::2], RG[2::2] = c * Gi[1::2] - s * Gi[2::2], s * Gi[1::2] + c * Gi[2::2]
    Z = torch.tensor(x["Z"], device=dev).reshape(2 * n, U)

    def back(z):                                  # samples (N, 2n, ...) -> rotated coefficients
        return torch.einsum("us,si...->iu...", RG, z)

    if call == "hypertime":
        zb = torch.tensor(x["z"], device=dev)
        V = torch.tensor(x["V"], device=dev)
        end, T = _integrate(case, m, w, zb, V.permute(1, 2, 0).contiguous(), dev)
        RT = G @ back(end).T - zb
        Jv = torch.einsum("su,iuk->ksi", G, back(T[:, :, :-1])) - V
        return {"RT": RT, "Jv": Jv}
    zb = G @ Z.T
    if call == "residual":
        return {"R": (back(_integrate(case, m, w, zb, None, dev)[0]) - Z).reshape(-1)}
    if call in ("jacobian", "products"):
        V = torch.tensor(x["V"], device=dev).reshape(-1, 2 * n, U)
        end, T = _integrate(case, m, w, zb, torch.einsum("su,kiu->sik", G, V).contiguous(), dev)
        R = (back(end) - Z).reshape(-1)
        Jv = (back(T[:, :, :-1]).permute(2, 0, 1) - V).reshape(V.shape[0], -1)
        if call == "products":
            return {"Jv": Jv}
        out = {"R": R, "Jv": Jv}
        if case["precision"] == "fp64":
            out["dRdw"] = back(T[:, :, -1]).reshape(-1)
        return out
    eye = torch.eye(2 * n, device=dev, dtype=torch.float64).expand(N, 2 * n, 2 * n)
    end, T = _integrate(case, m, w, zb, eye, dev)
    Phi = T[:, :, :-1]
    if call == "lyapunov":
        d = torch.ones(2 * n, device=dev, dtype=torch.float64)
        d[n:] = w
        Psi = d[:, None] * Phi / d
        Q = torch.eye(2 * n, case["h"], device=dev, dtype=torch.float64)
        acc = torch.zeros(case["h"], device=dev, dtype=torch.float64)
        kt = torch.tensor(_harmonics(case), device=dev, dtype=torch.float64)
        rho = torch.tensor(RHO[3 if case["s3"] else 2], device=dev, dtype=torch.float64)
        for i in range(case["n_ly"]):
            arg = kt @ (2 * math.pi * i * rho)
            H = torch.ones(U, device=dev, dtype=torch.float64)
            H[1::2], H[2::2] = torch.cos(arg), torch.sin(arg)
            A = torch.einsum("s,sij,jc->ic", H @ Gi, Psi, Q)
            Q, Rr = torch.linalg.qr(A)
            sg = torch.sign(torch.diagonal(Rr))
            Q = Q * sg
            acc += torch.log(torch.diagonal(Rr).abs())
        return {"sigma": acc * w / (2 * math.pi * case["n_ly"])}
    R = back(end) - Z
    res = float(torch.linalg.norm(R))
    if 2 * n * U <= 6000:
        J = torch.einsum("us,sij,sv->iujv", RG, Phi, G).reshape(2 * n * U, 2 * n * U)
        dZ = torch.linalg.solve(J - torch.eye(2 * n * U, device=dev, dtype=torch.float64), -R.reshape(-1))
    else:
        dZ = _gmres(lambda v: (back(torch.einsum("sij,sj->si", Phi, G @ v.reshape(2 * n, U).T)) - v.reshape(2 * n, U))
                    .reshape(-1), -R.reshape(-1), 400)
    return {"Z": Z.reshape(-1) + dZ, "res": torch.tensor(res, dtype=torch.float64)}


def _gmres(A, b, most):
    """Full GMRES to 1e-13 (modified Gram-Schmidt twice)."""
    beta = torch.linalg.norm(b)
    Q = [b / beta]
    H = np.zeros((most + 1, most))
    y = None
    for k in range(most):
        v = A(Q[k])
        B = torch.stack(Q)
        for _ in range(2):
            c = B @ v
            v = v - c @ B
            H[:k + 1, k] += c.cpu().numpy()
        H[k + 1, k] = float(torch.linalg.norm(v))
        e = np.zeros(k + 2)
        e[0] = float(beta)
        y, *_ = np.linalg.lstsq(H[:k + 2, :k + 1], e, rcond=None)
        if np.linalg.norm(H[:k + 2, :k + 1] @ y - e) <= 1e-13 * float(beta) or H[k + 1, k] == 0:
            break
        Q.append(v / H[k + 1, k])
    return torch.tensor(y, device=b.device) @ torch.stack(Q[:len(y)])
