"""The work that users of this framework have it do, as cases for timing and for comparing results.

A case names one call of the package's public entry points on a cubed-sphere shell (n x n cells on
each of six panels, n_r radial layers, degree p) or on rows of closure samples.  `prepare` makes what
the caller has in hand (the mesh handle, the prepared background, a seeded state, the workspace),
`run` is the call, `work` the bytes and operations it cannot do without, and `exact` the same result
from plain torch in 64 bits.
"""
import functools
import math

import numpy as np
import torch

from chorus_inputs import HEX20_REF2, BatchConfig, ShellConfig, cubed_sphere_hex20, make_phys, paper_case_phys
from paper_1503_00834_gb300 import FP32_PERT, FP64, Shell, Shells
from paper_1503_00834_gb300 import native

DEV = "cuda"
AMP = 1e-3  # relative size of the seeded perturbation, as in the shell workloads

# SSP-RK3 in Shu-Osher form: u_new = a u^n + b (u_k + dt L(u_k)) for each stage's (a, b)
SSPRK3 = ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))


def listed():
    return [
        # one residual of the smallest shell of the workloads (288 elements): four launches, all latency
        dict(name="residual_288_p3", kind="residual", n=4, n_r=3, p=3, phys="shell", prec="fp32"),
        # ten SSP-RK3 steps of a small odd-sized shell, as in a parameter study: launch bound
        dict(name="steps10_1470_p3", kind="step", n=7, n_r=5, p=3, phys="shell", prec="fp32", steps=10),
        # the headline workload: one SSP-RK3 step of the 331,776-element p = 3 shell
        dict(name="step_331776_p3", kind="step", n=48, n_r=24, p=3, phys="shell", prec="fp32", steps=1),
        # the coarse shell that the closure work steps
        dict(name="step_98304_p2", kind="step", n=32, n_r=16, p=2, phys="shell", prec="fp32", steps=1),
        # p = 4, the solar workload's order, odd sizes
        dict(name="step_111078_p4", kind="step", n=33, n_r=17, p=4, phys="shell", prec="fp32", steps=1),
        # the fine shell that the closure's pairs come from
        dict(name="step_98304_p5", kind="step", n=32, n_r=16, p=5, phys="shell", prec="fp32", steps=1),
        # the total-state form in double precision
        dict(name="step_fp64_24000_p3", kind="step", n=20, n_r=10, p=3, phys="shell", prec="fp64", steps=1),
        # a production step of the solar set: SSP-RK(5,4), radial kappa_r, diagnostics, angular-momentum correction
        dict(name="production_38016_p3_sun", kind="production", n=24, n_r=11, p=3, phys="sun", prec="fp32"),
        # an ensemble of independent shells of mixed order advanced together
        dict(name="batch_16", kind="batch", shells=16, n_lo=8, n_hi=16, nr_lo=4, nr_hi=8, steps=4),
        # a coarse shell with the learned closure attached
        dict(name="closure_step_41472_p2", kind="closure_step", n=24, n_r=12),
        # one gradient of the closure's training on a few batches' worth of samples
        dict(name="closure_grad_8192", kind="closure_grad", rows=8192),
        # a step of a state that lives in host memory, end to end
        dict(name="host_step_98304_p3", kind="host_step", n=32, n_r=16, p=3, phys="shell", prec="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "step", "step", "step", "step", "step64", "production", "batch", "closure_step",
                       "closure_grad", "host_step"])
    p = rng.choice([2, 3, 3, 4, 5])
    n, n_r = _log(rng, 3, 40), _log(rng, 2, 20)
    while 6 * n * n * n_r * (p + 1) ** 3 > 15_000_000:  # no more work than the largest listed case
        n -= 1
    phys = rng.choice(["shell", "shell", "sun"])
    if kind == "residual":
        return dict(kind=kind, n=n, n_r=n_r, p=p, phys=phys, prec=rng.choice(["fp32", "fp32", "fp64"]))
    if kind == "step":
        return dict(kind=kind, n=n, n_r=n_r, p=p, phys=phys, prec="fp32", steps=10 if n * n * n_r < 500 else 1)
    if kind == "step64":
        return dict(kind="step", n=min(n, 20), n_r=min(n_r, 10), p=p, phys=phys, prec="fp64", steps=1)
    if kind == "production":
        return dict(kind=kind, n=min(n, 30), n_r=n_r, p=p, phys=phys, prec="fp32")
    if kind == "batch":
        lo = _log(rng, 3, 10)
        return dict(kind=kind, shells=rng.randint(3, 16), n_lo=lo, n_hi=lo + rng.randint(1, 7), nr_lo=2, nr_hi=rng.randint(3, 8),
                    steps=rng.randint(1, 4))
    if kind == "closure_step":
        return dict(kind=kind, n=n, n_r=n_r)
    if kind == "closure_grad":
        return dict(kind=kind, rows=_log(rng, 100, 40000))
    return dict(kind=kind, n=min(n, 32), n_r=n_r, p=p, phys=phys, prec="fp32")


# ---------------------------------------------------------------- what a program has in hand


def _config(n, n_r, p, phys):
    if phys == "sun":
        beta, ph = paper_case_phys("sun")
    else:
        beta, ph = 0.75, make_phys(0.75, 1.5, 3.0, 1e-3)
    return ShellConfig("shell", n, n_r, p, beta, 1.0, 1, AMP, 1, ph)


def _shape20(xi, eta, zeta):
    """The 20 serendipity shape functions at broadcast reference points of [0,1]^3: [..., 20]."""
    a, b, c = np.broadcast_arrays(2.0 * xi - 1.0, 2.0 * eta - 1.0, 2.0 * zeta - 1.0)
    out = []
    for ai, bi, ci in HEX20_REF2 - 1.0:
        fa = 1 - a * a if ai == 0 else 1 + a * ai
        fb = 1 - b * b if bi == 0 else 1 + b * bi
        fc = 1 - c * c if ci == 0 else 1 + c * ci
        corner = ai != 0 and bi != 0 and ci != 0
        out.append(0.125 * fa * fb * fc * (a * ai + b * bi + c * ci - 2.0) if corner else 0.25 * fa * fb * fc)
    return np.stack(out, axis=-1)


def _points(N):
    """Solution points (Chebyshev-Gauss) and flux points (0, the Legendre-Gauss points, 1) on [0,1]."""
    xs = 0.5 * (1.0 - np.cos((2.0 * np.arange(1, N + 1) - 1.0) / (2.0 * N) * np.pi))
    xf = np.concatenate([[0.0], 0.5 * (np.polynomial.legendre.leggauss(N - 1)[0] + 1.0), [1.0]])
    return xs, xf


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


@functools.lru_cache(maxsize=24)
def _nodes(n, n_r, beta):
    xyz, h20 = cubed_sphere_hex20(n, n_r, beta, 1.0)
    return _t(xyz[h20]), _t(h20)


def _polytrope(phys, beta):
    """Constants of rho_a = rho_c chi^n, p_a = p_c chi^(n+1), chi = c + alpha d / r."""
    d, m = 1.0 - beta, phys.poly_n
    chi_o = (beta + 1.0) / (beta * math.exp(phys.N_rho / m) + 1.0)
    c = (2.0 * chi_o - beta - 1.0) / (1.0 - beta)
    alpha = (1.0 + beta) * (1.0 - chi_o) / (1.0 - beta) ** 2
    return c, alpha * d, phys.GM * phys.rho_c / ((m + 1.0) * alpha * d)


def _background(cfg):
    """x [E,3,N,N,N] and the polytrope's rho, E at the solution points."""
    xs, _ = _points(cfg.p + 1)
    nodes, _ = _nodes(cfg.n, cfg.n_r, cfg.r_inner)
    x = torch.einsum("kjia,eac->eckji", _t(_shape20(xs[None, None, :], xs[None, :, None], xs[:, None, None])), nodes)
    c, ad, p_c = _polytrope(cfg.phys, cfg.r_inner)
    chi = c + ad / x.square().sum(1).sqrt()
    return x, cfg.phys.rho_c * chi ** cfg.phys.poly_n, p_c * chi ** (cfg.phys.poly_n + 1.0) / (cfg.phys.gamma - 1.0)


@functools.lru_cache(maxsize=24)
def _density(n, n_r, p, phys):
    _, rho, en = _background(_config(n, n_r, p, phys))
    return rho.flatten(1).float(), en.flatten(1).float()


def _perturbation(n, n_r, p, phys, seed):
    """q' = Q - Q0 [E,5,N^3] FP32: entropy and pressure noise at every point, velocities of the same relative size."""
    rho, en = _density(n, n_r, p, phys)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    xi = torch.rand((rho.shape[0], 5, rho.shape[1]), generator=g, device=DEV).mul_(2.0).sub_(1.0)
    q = torch.empty_like(xi)
    q[:, 0] = rho * torch.expm1(-AMP * xi[:, 0])
    q[:, 1:4] = rho[:, None] * (0.3 * AMP) * xi[:, 1:4]
    q[:, 4] = en * (0.1 * AMP) * xi[:, 4]
    return q


@functools.lru_cache(maxsize=24)
def _shell(n, n_r, p, phys, use=""):
    """The mesh handle with its prepared background, kept by a program for all its states.  `use`: a
    handle of its own for calls that change the mesh's settings (an attached closure)."""
    sh = Shell(_config(n, n_r, p, phys))
    sh.mesh.prepare(sh.params)
    return sh


def _batch_config(case):
    return BatchConfig("batch", case["shells"], 4, case["n_lo"], case["n_hi"], case["nr_lo"], case["nr_hi"], (2, 3, 4, 5),
                       0.75, 1.0, AMP, make_phys(0.75, 1.5, 3.0, 1e-3))


@functools.lru_cache(maxsize=4)
def _shells(key):
    return Shells(_batch_config(dict(key)))


def _closure_params(seed, scale_out):
    """Seeded network: BF16 weights, FP32 biases and scales."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def u(shape, lim):
        return (torch.rand(shape, generator=g, device=DEV) * 2.0 - 1.0) * lim

    W = [u((128, 135), math.sqrt(3.0 / 135)).bfloat16(), u((128, 128), math.sqrt(3.0 / 128)).bfloat16(),
         u((135, 128), 0.1 * math.sqrt(3.0 / 128)).bfloat16()]
    b = [u((128,), 0.1), u((128,), 0.1), u((135,), 0.01)]
    ins = torch.tensor([AMP, AMP, AMP, AMP, AMP], device=DEV)
    outs = torch.tensor([scale_out] * 5, device=DEV)
    return W, b, ins, outs


def _closure_record(W, b, ins, outs):
    """The record of chorus_closure_bytes(): W1, W2, W3 BF16, then b1, b2, b3, the two scales FP32."""
    rec = torch.zeros(int(native.load().chorus_closure_bytes()), dtype=torch.uint8, device=DEV)
    data = torch.cat([w.reshape(-1).view(torch.uint8) for w in W]
                     + [v.float().contiguous().view(torch.uint8) for v in (*b, ins, outs)])
    rec[:data.numel()] = data
    return rec


def _closure_rows(rows, seed):
    """Samples as the pairs of a run have them: inputs of order one, targets of the same size."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 7)
    X = torch.rand((rows, 135), generator=g, device=DEV) * 2.0 - 1.0
    return X, torch.tanh(X.roll(3, 1)) * 0.5 + 0.1 * torch.rand((rows, 135), generator=g, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "closure_grad":
        X, Y = _closure_rows(case["rows"], seed)
        rec = _closure_record(*_closure_params(seed, 1.0))
        return dict(kind=kind, w=rec, X=X, Y=Y, grad=torch.empty(native.N_PARAMS, device=DEV))
    if kind == "batch":
        key = tuple(sorted((k, v) for k, v in case.items() if k not in ("kind", "name", "steps")))
        sh = _shells(key)
        Q = torch.zeros(sh.batch.n_state, device=DEV)
        for s, c in enumerate(sh.cfgs):
            sh.batch.view(Q, s).copy_(_perturbation(c.n, c.n_r, c.p, "shell", seed * 1000 + s))
        ws = torch.empty(sh.batch.workspace_bytes, dtype=torch.uint8, device=DEV)
        return dict(kind=kind, sh=sh, Q=Q, ws=ws, steps=case["steps"])
    if kind == "closure_step":
        sh = _shell(case["n"], case["n_r"], 2, "shell", "closure")
        q = _perturbation(case["n"], case["n_r"], 2, "shell", seed)
        ws = torch.empty(sh.mesh.workspace_bytes(FP32_PERT), dtype=torch.uint8, device=DEV)
        return dict(kind=kind, sh=sh, Q=q, ws=ws, w=_closure_record(*_closure_params(seed, 1e-2)))
    sh = _shell(case["n"], case["n_r"], case["p"], case["phys"])
    prec = FP64 if case["prec"] == "fp64" else FP32_PERT
    q = _perturbation(case["n"], case["n_r"], case["p"], case["phys"], seed)
    if prec == FP64:
        q = _total(_config(case["n"], case["n_r"], case["p"], case["phys"]), q)
    st = dict(kind=kind, sh=sh, prec=prec, ws=torch.empty(sh.mesh.workspace_bytes(prec), dtype=torch.uint8, device=DEV))
    if kind == "host_step":
        st["host"] = q.cpu().pin_memory()
        st["Q"] = torch.empty_like(q)
    else:
        st["Q"] = q
    if kind == "residual":
        st["R"] = torch.empty_like(q)
    st["steps"] = case.get("steps", 1)
    return st


def _total(cfg, q):
    """The total state Q0 + q' in double precision, [E,5,N^3]."""
    _, rho, en = _background(cfg)
    Q = q.double()
    Q[:, 0] += rho.flatten(1)
    Q[:, 4] += en.flatten(1)
    return Q.contiguous()


# ---------------------------------------------------------------- the calls


def run(s):
    kind = s["kind"]
    if kind == "closure_grad":
        return dict(loss=native.closure_grad(s["w"], s["X"], s["Y"], s["grad"]), grad=s["grad"])
    sh = s["sh"]
    if kind == "batch":
        sh.batch.rk_step(s["Q"], s["ws"], sh.dt, s["steps"])
        return s["Q"]
    if kind == "closure_step":
        native.closure_attach(sh.mesh, s["w"])
        sh.mesh.rk_step(sh.params, FP32_PERT, s["Q"], s["ws"], sh.dt, 1)
        return s["Q"]
    if kind == "residual":
        sh.mesh.residual(sh.params, s["prec"], s["Q"], s["R"], s["ws"])
        return s["R"]
    if kind == "step":
        sh.mesh.rk_step(sh.params, s["prec"], s["Q"], s["ws"], sh.dt, s["steps"])
        return s["Q"]
    if kind == "host_step":
        sh.mesh.rk_step_host(sh.params, s["prec"], s["host"], s["Q"], s["ws"], sh.dt, 1)
        return s["host"]
    # production: a step of the paper's integrator, the run's diagnostics, the angular-momentum correction
    sh.mesh.rk_step_scheme(sh.params, s["prec"], 1, s["Q"], s["ws"], sh.dt, 1)
    sums = sh.mesh.reduce(sh.params, s["prec"], s["Q"])
    return dict(sums=sums, domega=sh.mesh.am_correct(sh.params, s["prec"], s["Q"]), Q=s["Q"])


# ---------------------------------------------------------------- what a call cannot do without


def _stage_work(elems, p, stages, extra_reads, word):
    """Bytes and operations of `stages` residual evaluations: each stage needs the whole previous stage,
    so it reads its state, writes a new one (`extra_reads` stages also read the step's start) and
    reads the metrics (a row of three per flux point, |J|); per flux point of the three directions
    the state, the gradients and the fluxes, per solution point the derivatives."""
    N = p + 1
    dof, flux = N ** 3, 3 * (N + 1) * N * N
    words = stages * (10 * dof + 3 * flux + dof) + extra_reads * 5 * dof
    flops = stages * (flux * (17 * 2 * N + 200) + dof * (3 * 5 * 4 * (N + 1) + 250))
    return elems * words * word, elems * flops


def work(case):
    kind = case["kind"]
    if kind == "closure_grad":
        n = case["rows"]
        params = 128 * 135 + 128 * 128 + 135 * 128
        return dict(bytes=n * 270 * 4 + params * 6, flops=6 * n * params)
    if kind == "batch":
        k = case["steps"]
        each = [_stage_work(c.n_elem, c.p, 3 * k, 2 * k, 4) for c in _batch_config(case).shells()]
        return dict(bytes=sum(b for b, _ in each), flops=sum(f for _, f in each))
    elems = 6 * case["n"] ** 2 * case["n_r"]
    if kind == "closure_step":
        b, f = _stage_work(elems, 2, 3, 2, 4)
        return dict(bytes=b + 105000, flops=f + 3 * elems * 2 * (128 * 135 + 128 * 128 + 135 * 128))
    word = 8 if case["prec"] == "fp64" else 4
    if kind == "residual":
        b, f = _stage_work(elems, case["p"], 1, 0, word)
    elif kind == "production":
        # stages 2 to 5 read an earlier state, stage 4 also writes a second one; the reduction and the
        # correction each read the state, the quadrature weights and the coordinates
        b, f = _stage_work(elems, case["p"], 5, 6, word)
        dof = elems * (case["p"] + 1) ** 3
        b, f = b + dof * (3 * 5 * word + 2 * 4 * 8), f + dof * 80
    else:
        b, f = _stage_work(elems, case["p"], 3 * case.get("steps", 1), 2 * case.get("steps", 1), word)
        if kind == "host_step":  # the state in from the host and back
            b += 2 * elems * 5 * (case["p"] + 1) ** 3 * word
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- the same results in plain torch, 64 bits


def _lagrange(nodes, x):
    """Values and derivatives at x of the Lagrange basis through `nodes`: two [len(x), len(nodes)]."""
    n = len(nodes)
    val, der = np.ones((len(x), n)), np.zeros((len(x), n))
    for i in range(n):
        for s in range(n):
            if s != i:
                val[:, i] *= (x - nodes[s]) / (nodes[i] - nodes[s])
        for m in range(n):
            if m != i:
                t = np.full(len(x), 1.0 / (nodes[i] - nodes[m]))
                for s in range(n):
                    if s not in (i, m):
                        t = t * (x - nodes[s]) / (nodes[i] - nodes[s])
                der[:, i] += t
    return val, der


class _Discretization:
    """The spectral-difference residual of one shell in double precision.  Arrays along direction d
    are kept as lines, [..., t2, t1, s]: s along d, (t1, t2) the other two directions in order."""

    CORNERS = ((0, 3, 4, 7), (1, 2, 5, 6), (0, 1, 4, 5), (3, 2, 7, 6), (0, 1, 2, 3), (4, 5, 6, 7))  # (t1, t2) = 00, 10, 01, 11

    def __init__(self, cfg):
        self.cfg, self.ph, self.N = cfg, cfg.phys, cfg.p + 1
        N = self.N
        xs, xf = _points(N)
        I, _ = _lagrange(xs, xf)
        Lfs, D = _lagrange(xf, xs)
        _, Dff = _lagrange(xf, xf)
        self.I, self.D, self.Lfs = _t(I), _t(D), _t(Lfs)
        gx, gw = np.polynomial.legendre.leggauss(N)
        self.w = _t((0.5 * gw) @ _lagrange(xs, 0.5 * (gx + 1.0))[0])
        nodes, h20 = _nodes(cfg.n, cfg.n_r, cfg.r_inner)
        self.E = nodes.shape[0]
        self.x, self.rho0, self.en0 = _background(cfg)
        c, ad, p_c = _polytrope(self.ph, cfg.r_inner)
        T_a = p_c / (self.ph.R_gas * self.ph.rho_c) * (c + ad / cfg.r_outer)
        self.T_top = T_a if math.isnan(self.ph.T_top) else self.ph.T_top
        self._geometry(nodes, xf, Dff)
        self._faces(nodes, h20)
        r = self.x.square().sum(1).sqrt()
        kr = self.ph.kappa_r + (self.ph.kappa_r1 + self.ph.kappa_r2 * r) * r
        self.kr = [self.lines(kr, d) @ self.I.T for d in range(3)]
        self.gvec = -self.ph.GM * self.x / (r ** 3)[:, None]

    @staticmethod
    def lines(u, d):
        return u.movedim(-1 - d, -1)

    @staticmethod
    def points(u, d):
        return u.movedim(-1, -1 - d)

    def _geometry(self, nodes, xf, Dff):
        """Conservative curl-form metrics S^d at the flux points and |J| at the solution points, from
        coordinates about each element's centre."""
        N, E = self.N, self.E
        shp = _t(_shape20(xf[None, None, :], xf[None, :, None], xf[:, None, None]))
        Dff, L, Df = _t(Dff), self.Lfs, self.D
        self.S = [torch.empty((E, 3, N, N, N + 1), dtype=torch.float64, device=DEV) for _ in range(3)]
        self.detJ = torch.empty((E, N, N, N), dtype=torch.float64, device=DEV)
        for e0 in range(0, E, 32768):
            sl = slice(e0, min(E, e0 + 32768))
            nd = nodes[sl] - nodes[sl].mean(1, keepdim=True)
            X = torch.einsum("zyxa,eac->eczyx", shp, nd)
            dX = (X @ Dff.T, torch.einsum("by,eczyx->eczbx", Dff, X), torch.einsum("bz,eczyx->ecbyx", Dff, X))
            J = (torch.einsum("kz,jy,ix,eczyx->eckji", L, L, Df, X), torch.einsum("kz,jy,ix,eczyx->eckji", L, Df, L, X),
                 torch.einsum("kz,jy,ix,eczyx->eckji", Df, L, L, X))
            self.detJ[sl] = (J[0] * torch.linalg.cross(J[1], J[2], dim=1)).sum(1)
            for n in range(3):
                m, l = (n + 1) % 3, (n + 2) % 3
                V = [X[:, l] * dX[d][:, m] for d in range(3)]
                self.S[0][sl, n] = -(torch.einsum("jy,kz,ezyf->ekjf", Df, L, V[2]) - torch.einsum("jy,kz,ezyf->ekjf", L, Df, V[1]))
                self.S[1][sl, n] = -(torch.einsum("kz,ix,ezfx->ekif", Df, L, V[0]) - torch.einsum("kz,ix,ezfx->ekif", L, Df, V[2]))
                self.S[2][sl, n] = -(torch.einsum("ix,jy,efyx->ejif", Df, L, V[1]) - torch.einsum("ix,jy,efyx->ejif", L, Df, V[0]))

    def _faces(self, nodes, h20):
        """For each face its partner face (index 6 e + F, or -1 on a wall) and the partner's point of each point."""
        N, E = self.N, self.E
        cor = torch.stack([h20[:, list(c)] for c in self.CORNERS], 1).reshape(-1, 4)
        key = cor.sort(1).values
        key = (key[:, 0] << 42) + (key[:, 1] << 21) + key[:, 2]
        key, order = key.sort()
        same = (key[1:] == key[:-1]).nonzero()[:, 0]
        a, b = order[same], order[same + 1]
        self.nb = torch.full((E * 6,), -1, dtype=torch.int64, device=DEV)
        self.nb[a], self.nb[b] = b, a
        part = cor[self.nb.clamp(min=0)]
        p0 = (part == cor[:, :1]).to(torch.int64).argmax(1)
        p1 = (part == cor[:, 1:2]).to(torch.int64).argmax(1)
        table = np.zeros((4, 4, N * N), dtype=np.int64)
        for q0 in range(4):
            for q1 in range(4):
                s = np.array([(q1 & 1) - (q0 & 1), (q1 >> 1) - (q0 >> 1)])  # the partner's step along own t1
                if np.abs(s).sum() != 1:
                    continue
                for t in range(N * N):
                    pos = [0, 0]
                    for ax in range(2):
                        v = t % N if s[ax] != 0 else t // N
                        pos[ax] = N - 1 - v if (q0 >> ax) & 1 else v
                    table[q0, q1, t] = pos[0] + N * pos[1]
        self.perm = _t(table)[p0, p1]
        wall = (self.nb < 0).nonzero()[:, 0]
        self.wall = wall
        rad = nodes.reshape(-1, 3)[(wall // 6)[:, None] * 20 + torch.tensor(self.CORNERS, device=DEV)[wall % 6]].square().sum(-1).sqrt()
        self.top = ((rad.mean(1) - self.cfg.r_outer).abs() < (rad.mean(1) - self.cfg.r_inner).abs())[:, None]

    def ends(self, lines):
        """Values [E*6, ..., N^2] on the six faces of per-direction line arrays [E, ..., t2, t1, f]."""
        out = torch.stack([lines[F // 2][..., -1 if F % 2 else 0].flatten(-2) for F in range(6)], 1)
        return out.flatten(0, 1)

    def partner(self, v):
        """The partner faces' values at own points of [E*6, C, N^2]."""
        idx = self.perm[:, None, :].expand(-1, v.shape[1], -1)
        return torch.gather(v[self.nb.clamp(min=0)], 2, idx)

    def primitives(self, q):
        u = q[:, 1:4] / q[:, :1]
        return q[:, 0], u, (self.ph.gamma - 1.0) * (q[:, 4] - 0.5 * (q[:, 1:4] * u).sum(1))

    def inviscid(self, q, s):
        """s . (F, G, H) of [*, 5, ...] for directions s [*, 3, ...]."""
        _, u, p = self.primitives(q)
        vn = (u * s).sum(1)
        return torch.cat([(q[:, 1:4] * s).sum(1, keepdim=True), q[:, 1:4] * vn[:, None] + p[:, None] * s,
                          (vn * (q[:, 4] + p))[:, None]], 1)

    def heat(self, rho, p, g, kr, s):
        """s . f, f = -kappa rho T grad S - kappa_r rho C_p grad T; g [*, 5 (rho u v w p), 3, ...]."""
        A = (p / rho)[:, None] * g[:, 0]
        cpr = self.ph.gamma / (self.ph.gamma - 1.0)
        f = -cpr * (self.ph.kappa * (g[:, 4] / self.ph.gamma - A) + kr[:, None] * (g[:, 4] - A))
        return (f * s).sum(1)

    def traction(self, rho, g, s):
        """tau s of the trace-free stress with mu = rho nu."""
        gu = g[:, 1:4]
        div = gu[:, 0, 0] + gu[:, 1, 1] + gu[:, 2, 2]
        ts = (gu * s[:, None]).sum(2) + (gu * s[:, :, None]).sum(1) - (2.0 / 3.0) * div[:, None] * s
        return (rho * self.ph.nu)[:, None] * ts

    def viscous(self, q, g, kr, s):
        rho, u, p = self.primitives(q)
        ts = self.traction(rho, g, s)
        return torch.cat([torch.zeros_like(ts[:, :1]), ts, ((u * ts).sum(1) - self.heat(rho, p, g, kr, s))[:, None]], 1)

    def residual(self, Q):
        ph, N, E = self.ph, self.N, self.E
        Qf = [self.lines(Q, d) @ self.I.T for d in range(3)]
        own = self.ends(Qf)  # [E*6, 5, N^2]
        Sface = self.ends(self.S)  # [E*6, 3, N^2]
        sigma = torch.tensor([-1.0, 1.0] * 3, dtype=torch.float64, device=DEV).repeat(E)[:, None]
        mag = Sface.square().sum(1).sqrt()
        nh = Sface * (sigma / mag)[:, None]
        oth = self.partner(own)
        # lifting: common face states, wall states with no normal velocity and the wall's pressure
        com = 0.5 * (own + oth)
        w = self.wall
        rho, u, p = self.primitives(own[w])
        uc = u - (u * nh[w]).sum(1, keepdim=True) * nh[w]
        pc = torch.where(self.top, ph.R_gas * rho * self.T_top, p)
        com[w] = torch.cat([rho[:, None], rho[:, None] * uc, (pc / (ph.gamma - 1.0) + 0.5 * rho * uc.square().sum(1))[:, None]], 1)
        com = com.view(E, 6, 5, N, N)
        grad = 0.0
        for d in range(3):
            F = Qf[d].clone()
            F[..., 0], F[..., -1] = com[:, 2 * d], com[:, 2 * d + 1]
            gx = self.S[d] @ self.Lfs.T  # S^d at the solution points
            grad = grad + self.points((F @ self.D.T)[:, :, None] * gx[:, None], d)
        del com
        grad = grad / self.detJ[:, None, None]  # [E, 5, 3, ...] conserved gradients
        rho, u, _ = self.primitives(Q)
        gr = grad[:, 0].clone()
        gp = (ph.gamma - 1.0) * (grad[:, 4] - (u[:, :, None] * grad[:, 1:4]).sum(1) + 0.5 * u.square().sum(1)[:, None] * gr)
        grad[:, 1:4] = (grad[:, 1:4] - u[:, :, None] * gr[:, None]) / rho[:, None, None]
        grad[:, 4] = gp
        # fluxes at the flux points, common fluxes at the faces
        G = [self.lines(grad, d) @ self.I.T for d in range(3)]
        del grad
        gf = self.ends(G)  # [E*6, 5, 3, N^2]
        krf = self.ends(self.kr)  # [E*6, N^2]
        Fv = self.viscous(own, gf, krf, nh)
        c = [(nh * v).sum(1).abs() + (ph.gamma * q / r).sqrt() for r, v, q in (self.primitives(own), self.primitives(oth))]
        Fn = 0.5 * (self.inviscid(own, nh) + self.inviscid(oth, nh)) - 0.5 * torch.maximum(*c)[:, None] * (oth - own)
        Fn = Fn - 0.5 * (Fv - self.partner(Fv))
        rho, u, p = self.primitives(own[w])
        trac = (self.traction(rho, gf[w], nh[w]) * nh[w]).sum(1)
        top = self.heat(rho, ph.R_gas * rho * self.T_top, gf[w], krf[w], nh[w])
        Fn[w] = torch.cat([torch.zeros_like(rho)[:, None], (p - trac)[:, None] * nh[w],
                           torch.where(self.top, top, torch.full_like(top, -ph.bottom_flux))[:, None]], 1)
        Fn = (Fn * (sigma * mag)[:, None]).view(E, 6, 5, N, N)
        del gf, Fv, oth
        div = 0.0
        for d in range(3):
            F = self.inviscid(Qf[d], self.S[d]) - self.viscous(Qf[d], G[d], self.kr[d], self.S[d])
            F[..., 0], F[..., -1] = Fn[:, 2 * d], Fn[:, 2 * d + 1]
            div = div + self.points(F @ self.D.T, d)
            Qf[d] = G[d] = None
        R = -div / self.detJ[:, None]
        R[:, 1:4] += Q[:, :1] * self.gvec
        R[:, 1] += 2.0 * ph.Omega * Q[:, 2]
        R[:, 2] -= 2.0 * ph.Omega * Q[:, 1]
        R[:, 4] += (Q[:, 1:4] * self.gvec).sum(1)
        return R

    def total(self, q):
        """The total state of a perturbation [E, 5, N^3]."""
        Q = q.double().view(self.E, 5, self.N, self.N, self.N).clone()
        Q[:, 0] += self.rho0
        Q[:, 4] += self.en0
        return Q

    def perturbation(self, Q):
        Q = Q.clone()
        Q[:, 0] -= self.rho0
        Q[:, 4] -= self.en0
        return Q.flatten(2)


def _rk3(L, u, dt, steps):
    for _ in range(steps):
        s = u
        for a, b in SSPRK3:
            s = a * u + b * (s + dt * L(s))
        u = s
    return u


def _rk54(L, u, dt):
    """SSP-RK(5,4) of Spiteri and Ruuth, published coefficients."""
    u1 = u + 0.391752226571890 * dt * L(u)
    u2 = 0.444370493651235 * u + 0.555629506348765 * u1 + 0.368410593050371 * dt * L(u1)
    u3 = 0.620101851488403 * u + 0.379898148511597 * u2 + 0.251891774271694 * dt * L(u2)
    L3 = L(u3)
    u4 = 0.178079954393132 * u + 0.821920045606868 * u3 + 0.544974750228521 * dt * L3
    return (0.517231671970585 * u2 + 0.096059710526147 * u3 + 0.063692468666290 * dt * L3 + 0.386708617503269 * u4
            + 0.226007483236906 * dt * L(u4))


def _network(W, b, X, rounded):
    """The closure network on rows X; `rounded`: each layer's input rounded to BF16, as its use in the
    stages is defined.  Returns the pre-activations and the output."""
    r = (lambda v: v.float().bfloat16().double()) if rounded else (lambda v: v)
    W, b = [w.double() for w in W], [v.double() for v in b]
    silu = torch.nn.functional.silu
    z1 = r(X) @ W[0].T + b[0]
    z2 = r(silu(z1)) @ W[1].T + b[1]
    return z1, z2, r(silu(z2)) @ W[2].T + b[2]


def _exact_grad(case, seed):
    W, b, _, _ = _closure_params(seed, 1.0)
    X, Y = (v.double() for v in _closure_rows(case["rows"], seed))
    z1, z2, y = _network(W, b, X, False)
    W = [w.double() for w in W]
    silu = torch.nn.functional.silu

    def slope(z):
        s = torch.sigmoid(z)
        return s * (1.0 + z * (1.0 - s))

    dy = (y - Y) / y.numel()
    d2 = (dy @ W[2]) * slope(z2)
    d1 = (d2 @ W[1]) * slope(z1)
    grads = [d1.T @ X, d2.T @ silu(z1), dy.T @ silu(z2), d1.sum(0), d2.sum(0), dy.sum(0)]
    return dict(loss=0.5 * float(((y - Y) ** 2).mean()), grad=torch.cat([g.reshape(-1) for g in grads]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "closure_grad":
        return _exact_grad(case, seed)
    if kind == "batch":
        sh = _shells(tuple(sorted((k, v) for k, v in case.items() if k not in ("kind", "name", "steps"))))
        out = torch.zeros(sh.batch.n_state, dtype=torch.float64, device=DEV)
        for s, c in enumerate(sh.cfgs):
            D = _Discretization(c)
            u = _rk3(D.residual, D.total(_perturbation(c.n, c.n_r, c.p, "shell", seed * 1000 + s)), sh.dt, case["steps"])
            sh.batch.view(out, s).copy_(D.perturbation(u))
        return out
    p, phys = case.get("p", 2), case.get("phys", "shell")
    D = _Discretization(_config(case["n"], case["n_r"], p, phys))
    dt = _shell(case["n"], case["n_r"], p, phys).dt
    q = _perturbation(case["n"], case["n_r"], p, phys, seed)
    if kind == "closure_step":
        W, b, ins, outs = _closure_params(seed, 1e-2)

        def L(Q):
            X = (D.perturbation(Q) / ins.double()[:, None]).flatten(1)
            return D.residual(Q) + (_network(W, b, X, True)[2].view(-1, 5, 27) * outs.double()[:, None]).view(Q.shape)

        return D.perturbation(_rk3(L, D.total(q), dt, 1))
    if case["prec"] == "fp64":
        u = _total(D.cfg, q).view(D.E, 5, D.N, D.N, D.N)
    else:
        u = D.total(q)
    if kind == "residual":
        return D.residual(u).flatten(2)
    if kind in ("step", "host_step"):
        u = _rk3(D.residual, u, dt, case.get("steps", 1))
        return u.flatten(2) if case["prec"] == "fp64" else D.perturbation(u)
    u = _rk54(D.residual, u, dt)
    wJ = D.detJ * D.w[:, None, None] * D.w[:, None] * D.w
    x = D.x
    ke = 0.5 * u[:, 1:4].square().sum(1) / u[:, 0]
    ang = (torch.linalg.cross(x, u[:, 1:4], dim=1) * wJ[:, None]).sum((0, 2, 3, 4))
    sums = torch.stack([(wJ * u[:, 0]).sum(), (wJ * u[:, 4]).sum(), (wJ * ke).sum(), ang.square().sum().sqrt()])
    inertia = ((x.square().sum(1, keepdim=True) - x.square()) * (wJ * u[:, 0])[:, None]).sum((0, 2, 3, 4))
    dO = ang / inertia
    mn = u[:, 1:4] - u[:, :1] * torch.linalg.cross(dO.view(1, 3, 1, 1, 1).expand_as(x), x, dim=1)
    u[:, 4] += 0.5 * (mn.square().sum(1) - u[:, 1:4].square().sum(1)) / u[:, 0]
    u[:, 1:4] = mn
    return dict(sums=sums, domega=dO, Q=D.perturbation(u))
