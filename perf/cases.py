"""What a user of the library has it do, as cases that can be timed and checked.

    listed()            the cases; draw(rng) one more of the same ranges
    prepare(case, seed) inputs on the GPU, made from the seed, and the handles that a program keeps
    run(state)          one pass through the public entry points and its outputs
    work(case)          bytes and flops that the pass cannot do without
    exact(case, seed)   the outputs in 64 bits from plain torch, without the library

Gauge fields are quenched U(1) fields (Metropolis, hot start, on the GPU) at the beta and m0 of the repository's
configurations.  Hierarchies whose own numbers reach an output (V-cycles, level differences, the estimate) are set up
without bootstrap rounds, the library's default, which makes them a function of the field and the seed alone.  Mixed
solves run to 1e-12, as the parity tests do, so that outputs are fixed by the equations and not by the stopping rule.
"""
import math

import numpy as np
import torch

from paper_2303_11512_gb300 import api

DEV = "cuda"
C64, C128 = torch.complex64, torch.complex128
PREC = {"fp64": api.FP64, "fp32": api.FP32, "mixed": api.MIXED}
PHASE_STOCH, PHASE_SKETCH, PHASE_TESTVEC, PHASE_HUTCH = 0, 1, 2, 3
HUTCH_SAMPLES = 64


# ---------------------------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the fine operator as the benchmark's stencil figure takes it: 256 right-hand sides, far larger than L2
        dict(name="stencil_fp32_L512_r256", op="stencil", L=512, rhs=256, prec="fp32", beta=5.0, m0=-0.05),
        # the smallest call of the library: one FP64 operator application on the 16 x 16 lattice
        dict(name="stencil_fp64_L16_r1", op="stencil", L=16, rhs=1, prec="fp64", beta=3.0, m0=-0.05),
        # the preconditioner of the benchmark's solves: V(2,2), FP16 coarse operators, a sketch's 32 vectors
        dict(name="vcycle_fp16_L512_r32", op="vcycle", L=512, rhs=32, prec="fp32", images=3, sweeps=2, ntv=8,
             beta=5.0, m0=-0.05),
        # the same with the library's defaults (V(1,1), TF32) on a small lattice and a few odd right-hand sides
        dict(name="vcycle_tf32_L128_r5", op="vcycle", L=128, rhs=5, prec="fp32", images=2, sweeps=1, ntv=8, beta=3.0,
             m0=-0.08),
        # the method's main cost: a batch of mixed-precision solves on the benchmark's lattice and set-up
        dict(name="solve_mixed_L512_r32", op="solve", L=512, rhs=32, prec="mixed", images=3, sweeps=2, bootstrap=2,
             beta=5.0, m0=-0.06),
        # the plain FP64 form that the mixed one is compared with, 64 right-hand sides a launch
        dict(name="solve_fp64_L128_r64", op="solve", L=128, rhs=64, prec="fp64", images=2, sweeps=1, bootstrap=0,
             beta=3.0, m0=-0.08),
        # one stochastic batch of Algorithm 2 on a middle level: noise, level difference, projected samples
        dict(name="sample_L256_l1_r24", op="sample", L=256, rhs=24, level=1, d=16, images=2, sweeps=1, beta=3.0,
             m0=-0.08),
        # a new gauge field: the whole multigrid set-up, and one V-cycle through what it built
        dict(name="setup_L512", op="setup", L=512, rhs=8, images=3, sweeps=2, beta=5.0, m0=-0.05),
        # Algorithm 2 end to end: sketches of every level difference and the stochastic loop
        dict(name="estimate_L128", op="estimate", L=128, samples=64, d=32, k=2, images=3, sweeps=2, beta=3.0, m0=-0.08),
        # Algorithm 1 on the smallest configuration: unpreconditioned GMRES(30), bound by launches and host decisions
        dict(name="hutchinson_L16", op="hutchinson", L=16, samples=HUTCH_SAMPLES, beta=3.0, m0=-0.05),
        # the learned correction as FGMRES applies it
        dict(name="net_forward_L256_r16", op="net", L=256, rhs=16, channels=16, grad=False, beta=3.0),
        # one training batch: loss and gradient
        dict(name="net_train_L128_r32", op="net", L=128, rhs=32, channels=16, grad=True, beta=3.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["stencil", "vcycle", "vcycle", "solve", "solve", "sample", "setup", "estimate", "hutchinson", "net"])
    beta, m0 = rng.choice([3.0, 5.0]), rng.choice([-0.02, -0.05])
    if op == "stencil":
        L = 2 * _log_int(rng, 4, 512)
        prec = rng.choice(["fp32", "fp64"])
        most = 512 * 512 * 256 // (L * L) // (1 if prec == "fp32" else 2)
        return dict(op=op, L=L, rhs=_log_int(rng, 1, max(1, min(256, most))), prec=prec, beta=beta, m0=m0)
    if op == "hutchinson":
        return dict(op=op, L=rng.choice([16, 32]), samples=rng.randrange(9, HUTCH_SAMPLES + 1), beta=beta, m0=m0)
    if op == "net":
        L, grad = rng.choice([16, 32, 48, 64, 128, 256]), rng.random() < 0.5
        return dict(op=op, L=L, rhs=_log_int(rng, 1, min(64, 256 * 256 * (8 if grad else 16) // (L * L))),
                    channels=rng.choice([4, 8, 16]), grad=grad, beta=beta)
    images, sweeps = rng.choice([0, 1, 2, 3]), rng.choice([1, 2])
    if op == "setup":
        return dict(op=op, L=rng.choice([32, 64, 128, 192, 256]), rhs=rng.randrange(1, 9), images=images, sweeps=sweeps,
                    beta=beta, m0=m0)
    if op == "estimate":
        return dict(op=op, L=rng.choice([32, 64, 128]), samples=rng.randrange(10, 65), d=rng.choice([8, 16, 32]),
                    k=rng.choice([1, 2]), images=images, sweeps=sweeps, beta=beta, m0=m0)
    if op == "sample":
        L = rng.choice([64, 128, 256])
        return dict(op=op, L=L, rhs=_log_int(rng, 1, min(64, 256 * 256 * 24 // (L * L))), level=rng.choice([0, 1]),
                    d=rng.choice([0, 8, 16]), images=images, sweeps=sweeps, beta=beta, m0=m0)
    if op == "vcycle":
        L, prec = rng.choice([32, 64, 128, 192, 256, 512]), rng.choice(["fp32", "fp32", "fp64"])
        most = 512 * 512 * 32 // (L * L) // (1 if prec == "fp32" else 16)
        return dict(op=op, L=L, rhs=_log_int(rng, 1, max(1, min(256, most))), prec=prec, images=images, sweeps=sweeps,
                    ntv=rng.choice([8, 8, 8, 4]), beta=beta, m0=m0)
    L, prec = rng.choice([32, 64, 128, 256, 512]), rng.choice(["mixed", "mixed", "fp64"])
    most = 512 * 512 * 32 // (L * L) if prec == "mixed" else 128 * 128 * 64 // (L * L)
    return dict(op=op, L=L, rhs=_log_int(rng, 1, max(1, min(256, most))), prec=prec, images=images, sweeps=sweeps,
                bootstrap=rng.choice([0, 2]) if prec == "mixed" else 0, beta=beta, m0=m0)


# --------------------------------------------------------------------------------------------------------- inputs
def _generator(seed, what):
    return torch.Generator(device=DEV).manual_seed(1000003 * seed + what)


def _links(L, beta, seed, sweeps=30):
    """Links exp(i theta) of a quenched U(1) field: single-hit checkerboard Metropolis from a hot start."""
    g = _generator(seed, 1)
    th = (torch.rand((L, L, 2), generator=g, dtype=torch.float64, device=DEV) * 2 - 1) * math.pi
    odd = torch.arange(L, device=DEV) % 2
    for _ in range(sweeps):
        for mu in (0, 1):
            for parity in (0, 1):
                prop, acc = torch.rand((2, L, L), generator=g, dtype=torch.float64, device=DEV)
                prop = 2 * prop - 1
                a, b = th[..., 0], th[..., 1]
                P = a + b.roll(-1, 1) - a.roll(-1, 0) - b
                sign = 1 if mu == 0 else -1
                Q = P.roll(1, mu)
                dS = -beta * ((P + sign * prop).cos() - P.cos() + (Q - sign * prop).cos() - Q.cos())
                mine = odd[:, None] == parity if mu == 0 else odd[None, :] == parity
                th[..., mu] += torch.where(mine & (acc < torch.exp(-dS)), prop, torch.zeros_like(prop))
    return torch.polar(torch.ones_like(th), th).contiguous()


def _vectors(seed, rhs, n, dtype, what=2):
    """Complex Gaussian vectors of unit norm, as Krylov vectors and residuals are."""
    x = torch.randn((rhs, n), generator=_generator(seed, what), dtype=C128 if dtype == C128 else C64, device=DEV)
    return (x / torch.linalg.vector_norm(x, dim=1, keepdim=True)).contiguous()


def _net_params(channels, seed):
    r = np.random.default_rng([seed, 7])
    dims = [2, channels, channels, channels, 2]
    W = [(r.standard_normal((9, o, i)) + 1j * r.standard_normal((9, o, i))) / math.sqrt(18 * i)
         for i, o in zip(dims[:-1], dims[1:])]
    b = [0.02 * r.standard_normal(o) for o in dims[1:-1]]
    return W, b


def _mg_params(case):
    return dict(ntv=case.get("ntv", 8), pre_smooth=case["sweeps"], post_smooth=case["sweeps"],
                tensor_cores=case["images"], bootstrap=case.get("bootstrap", 0), seed=11)


def prepare(case, seed):
    op, L = case["op"], case["L"]
    s = dict(case=case, seed=seed, ctx=api.Context(), U=_links(L, case["beta"], seed))
    n = 2 * L * L
    if op == "stencil":
        dt = C64 if case["prec"] == "fp32" else C128
        s["x"] = _vectors(seed, case["rhs"], n, dt)
        s["y"] = torch.empty_like(s["x"])
        return s
    if op == "net":
        s["net"] = api.Net(s["ctx"], s["U"], L, 4, case["channels"])
        s["net"].set_params(api.pack_params(*_net_params(case["channels"], seed)))
        s["r"], s["e"] = _vectors(seed, case["rhs"], n, C64), _vectors(seed, case["rhs"], n, C64, 3)
        return s
    if op == "setup":
        s["b"] = _vectors(seed, case["rhs"], n, C128)
        return s
    if op == "hutchinson":
        s["h"] = api.mg_setup(s["ctx"], s["U"], L, case["m0"])
        return s
    s["h"] = h = api.mg_setup(s["ctx"], s["U"], L, case["m0"], **_mg_params(case))
    if op == "vcycle":
        s["b"] = _vectors(seed, case["rhs"], n, C64 if case["prec"] == "fp32" else C128)
        s["x"] = torch.empty_like(s["b"])
    elif op == "solve":
        s["b"] = api.mgmlmc_rademacher(s["ctx"], seed, 0, PHASE_HUTCH, 0, n, case["rhs"])
        s["x"] = torch.empty_like(s["b"])
    elif op == "sample":
        l = min(case["level"], h.levels - 2)
        s["level"], s["sketch"] = l, None
        if case["d"]:
            s["sketch"], _ = api.hutchpp_sketch_qr(s["ctx"], h, l, case["d"], 1, seed, form=api.REDUCED, tol=1e-12)
        s["z"] = torch.empty((case["rhs"], h.n[l]), dtype=C128, device=DEV)
        s["y"] = torch.empty_like(s["z"])
    return s


# ----------------------------------------------------------------------------------------------------------- run
def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "stencil":
        api.schwinger_apply(ctx, s["U"], case["L"], case["m0"], s["x"], s["y"], PREC[case["prec"]])
        return s["y"]
    if op == "vcycle":
        s["h"].vcycle(0, s["b"], s["x"], PREC[case["prec"]])
        return s["x"]
    if op == "solve":
        tol = 1e-12 if case["prec"] == "mixed" else 1e-10
        api.fgmres_batched(ctx, s["h"], 0, s["b"], s["x"], tol=tol, prec=PREC[case["prec"]])
        return s["x"]
    if op == "sample":
        api.mgmlmc_rademacher(ctx, s["seed"], s["level"], PHASE_STOCH, 0, s["z"].shape[1], case["rhs"], s["z"])
        api.mlmc_level_sample(ctx, s["h"], s["level"], s["z"], s["y"], tol=1e-12)
        return api.hutchpp_project(ctx, s["sketch"], s["z"], s["y"]), s["y"]
    if op == "setup":
        h = api.mg_setup(ctx, s["U"], case["L"], case["m0"], **_mg_params(case))
        x64 = torch.empty_like(s["b"])
        h.vcycle(0, s["b"], x64, api.FP64)
        b32 = s["b"].to(C64)
        x32 = torch.empty_like(b32)
        h.vcycle(0, b32, x32, api.FP32)
        return np.complex128(h.coarsest_trace()), x64, x32
    if op == "estimate":
        r = api.trace_estimate(ctx, s["h"], eps=1e-3, d=case["d"], k=case["k"], nrhs_first=8, seed=s["seed"],
                               min_samples=case["samples"], max_samples=case["samples"], keep_samples=case["samples"],
                               tol=1e-12)
        return (np.complex128(r["tau"]), r["sigma"], np.complex128(r["tau_L"]), np.array(r["tau_lr"]),
                np.stack(r["samples"]))
    if op == "hutchinson":
        r = api.hutchinson_estimate(ctx, s["h"], eps=1e-6, seed=s["seed"], min_samples=case["samples"],
                                    max_samples=case["samples"], keep_samples=case["samples"], precond=0, m=30,
                                    tol=1e-10, prec=api.FP64, maxit=20000)
        return np.complex128(r["tau"]), r["sigma"], r["samples"]
    if not case["grad"]:
        return s["net"].forward(s["r"])
    return s["net"].loss_grad(s["r"], s["e"])


# ---------------------------------------------------------------------------------------------------------- work
def _sides(L):
    out = [L]
    while out[-1] > 8 and out[-1] % 16 == 0:
        out.append(out[-1] // 4)
    return out


def work(case):
    """Inputs read once and outputs written once; flops: one application of the operators that the pass is made of."""
    op, L = case["op"], case["L"]
    V = float(L * L)
    rhs = float(case.get("rhs", case.get("samples", 1)))
    z = 8.0 if case.get("prec") == "fp32" else 16.0
    dof = 2.0 * case.get("ntv", 8)
    sides = _sides(L)
    coarse = sum(5.0 * dof * dof * v * v for v in sides[1:-1]) + (sides[-1] ** 2 * dof) ** 2
    prolong = sum((2 if i == 0 else dof) * dof / 2 * v * v for i, v in enumerate(sides[:-1]))
    if op == "stencil":
        return dict(bytes=rhs * V * 4 * z + 32 * V, flops=52 * rhs * V)
    if op == "net":
        c = case["channels"]
        return dict(bytes=rhs * V * (48 if case["grad"] else 32) + 32 * V,
                    flops=(3 if case["grad"] else 1) * 8 * 9 * (2 * c + 2 * c * c + 2 * c) * V * rhs)
    if op == "hutchinson":  # a Krylov space of at least sqrt(condition) ~ 30 vectors for each sample
        return dict(bytes=32 * V, flops=30 * 52 * V * rhs)
    cycle = 2 * case["sweeps"] * (52 + 8 * 64) * V + 8 * 2 * prolong + 8 * 2 * (case["sweeps"] + 1) * coarse
    if op == "setup":  # Galerkin products, block inverses and the dense inverse, beside the two V-cycles
        sweeps = 4 * 8 * (52 + 8 * 64) * V
        return dict(bytes=32 * V + rhs * V * 2 * 56,
                    flops=sweeps + 8 * 5 * prolong * dof + 8 * 32 ** 3 * V / 16 + 8 * (sides[-1] ** 2 * dof) ** 3
                    + 2 * rhs * cycle)
    if op == "vcycle":
        return dict(bytes=rhs * V * 4 * z + 32 * V, flops=rhs * cycle)
    if op == "estimate":
        return dict(bytes=32 * V, flops=(len(sides) - 1) * (rhs + (case["k"] + 1) * case["d"]) * 5 * cycle)
    if op == "sample":
        v = sides[min(case["level"], len(sides) - 2)]
        return dict(bytes=rhs * v * v * 16 * (2 if v == L else dof), flops=rhs * 5 * cycle * (v / L) ** 2)
    return dict(bytes=rhs * V * 64 + 32 * V, flops=rhs * 5 * cycle)


# --------------------------------------------------------------------------------------------------------- exact
def _mix64(z):
    """SplitMix64 finaliser on int64 tensors (two's complement words)."""
    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)
    z = (z ^ shr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ shr(z, 31)


def _signs(seed, level, phase, sample0, rhs, n):
    """+-1 streams [rhs, n] of the counter-based generator."""
    sample = torch.arange(rhs, dtype=torch.int64, device=DEV) + sample0
    key = _mix64(seed ^ _mix64((level << 56) | (phase << 48) | sample))
    i = torch.arange(1, n + 1, dtype=torch.int64, device=DEV)
    w = _mix64(key[:, None] + (0x9E3779B97F4A7C15 - (1 << 64)) * i)
    return torch.where(w < 0, -1.0, 1.0).to(torch.float64)


def _shift(x, f):
    """x(s + f) on fields [T, X, ...]; f: 0 self, 1 +x, 2 -x, 3 +t, 4 -t."""
    return x if f == 0 else x.roll(-1 if f in (1, 3) else 1, 1 if f <= 2 else 0)


class _Op:
    """5-point block operator A[T, X, f, d, d] on fields [T, X, d, r], with its SAP blocks."""

    def __init__(self, A, bs=0):
        self.A, self.L, self.d, self.bs = A, A.shape[0], A.shape[-1], bs
        if bs:
            L, d, nb = self.L, self.d, self.L // bs
            D = torch.zeros((nb, nb, bs * bs, d, bs * bs, d), dtype=C128, device=DEV)
            blocks = A.reshape(nb, bs, nb, bs, 5, d, d)
            for j in range(bs * bs):
                t, x = divmod(j, bs)
                for f, (dt, dx) in enumerate([(0, 0), (0, 1), (0, -1), (1, 0), (-1, 0)]):
                    if 0 <= t + dt < bs and 0 <= x + dx < bs:
                        D[:, :, j, :, (t + dt) * bs + x + dx, :] = blocks[:, t, :, x, f]
            m = bs * bs * d
            self.inv = torch.linalg.inv(D.reshape(nb, nb, m, m))
            par = torch.arange(nb, device=DEV)
            self.colour = (par[:, None] + par[None, :]) % 2

    def __call__(self, x):
        if self.d > 2:
            return sum(torch.matmul(self.A[:, :, f], _shift(x, f)) for f in range(5))
        y = torch.zeros_like(x)
        for f in range(5):
            xs = _shift(x, f)
            for i in range(2):
                for j in range(2):
                    if f or i == j:
                        y[:, :, i].addcmul_(self.A[:, :, f, i, j, None], xs[:, :, j])
        return y

    def sweep(self, f, x):
        nb, bs, d, r = self.L // self.bs, self.bs, self.d, x.shape[-1]
        for c in (0, 1):
            res = (f - self(x)).reshape(nb, bs, nb, bs, d, r).transpose(1, 2).reshape(nb, nb, bs * bs * d, r)
            e = torch.matmul(self.inv, res) * (self.colour == c)[:, :, None, None]
            x = x + e.reshape(nb, nb, bs, bs, d, r).transpose(1, 2).reshape(x.shape)
        return x


def _fine(U, m0, bs=0):
    L = U.shape[0]
    W = -0.5 * U
    W[L - 1, :, 1] *= -1
    A = torch.zeros((L, L, 5, 2, 2), dtype=C128, device=DEV)
    eye = torch.eye(2, dtype=C128, device=DEV)
    A[:, :, 0] = (m0 + 2) * eye
    for mu, sig in enumerate([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]]]):
        sig = torch.tensor(sig, dtype=C128, device=DEV)
        A[:, :, 1 + 2 * mu] = W[:, :, mu, None, None] * (eye - sig)
        A[:, :, 2 + 2 * mu] = W[:, :, mu].roll(1, 1 - mu).conj()[:, :, None, None] * (eye + sig)
    return _Op(A, bs)


class _Multigrid:
    """The aggregation hierarchy of the library's default set-up, and what is computed with it."""

    def __init__(self, U, m0, ntv=8, pre=1, seed=11, setup_sweeps=4, agg=4):
        self.D, self.P, self.pre, self.agg = [_fine(U, m0, 4)], [], pre, agg
        sides = _sides(U.shape[0])
        for l, L in enumerate(sides[:-1]):
            D, d, Lc = self.D[l], self.D[l].d, L // agg
            hd = d // 2
            v = _signs(seed, l, PHASE_TESTVEC, 0, ntv, 2 * L * L * d).reshape(ntv, L, L, d, 2)
            v = torch.view_as_complex(v).permute(1, 2, 3, 0).contiguous()
            for _ in range(setup_sweeps):
                v = D.sweep(torch.zeros_like(v), v)
            B = v.reshape(Lc, agg, Lc, agg, 2, hd, ntv).permute(0, 2, 4, 1, 3, 5, 6)  # [T, X, c, jt, jx, k, m]
            Q, R = torch.linalg.qr(B.reshape(Lc, Lc, 2, agg * agg * hd, ntv))
            ph = R.diagonal(dim1=-2, dim2=-1)
            Q = (Q * (ph / ph.abs())[..., None, :]).reshape(Lc, Lc, 2, agg, agg, hd, ntv)
            P = torch.zeros((Lc, agg, Lc, agg, 2, hd, 2, ntv), dtype=C128, device=DEV)
            for c in (0, 1):
                P[:, :, :, :, c, :, c] = Q[:, :, c].permute(0, 2, 1, 3, 4, 5)
            P = P.reshape(L, L, d, 2 * ntv)  # fine site's rows of its aggregate's prolongator
            A = torch.zeros((Lc, Lc, 5, 2 * ntv, 2 * ntv), dtype=C128, device=DEV)
            at = torch.arange(L, device=DEV)
            for f in range(5):
                g = torch.matmul(P.mH, torch.matmul(D.A[:, :, f], _shift(P, f)))
                if f == 0:
                    out = torch.zeros((L, L, 1, 1), dtype=torch.bool, device=DEV)
                else:
                    edge = at % agg == (agg - 1 if f in (1, 3) else 0)
                    out = (edge[None, :] if f <= 2 else edge[:, None]).expand(L, L)[:, :, None, None]
                for to, part in ((0, g * ~out), (f, g * out)):
                    A[:, :, to] += part.reshape(Lc, agg, Lc, agg, 2 * ntv, 2 * ntv).sum((1, 3))
            self.P.append(P)
            self.D.append(_Op(A, 2 if l + 2 < len(sides) else 0))
        last = self.D[-1]
        m = last.L * last.L * last.d
        unit = torch.eye(m, dtype=C128, device=DEV).reshape(last.L, last.L, last.d, m)
        self.inv = torch.linalg.inv(last(unit).reshape(m, m))

    def restrict(self, l, x):
        a, Lc = self.agg, self.D[l].L // self.agg
        y = torch.matmul(self.P[l].mH, x)
        return y.reshape(Lc, a, Lc, a, *y.shape[2:]).sum((1, 3))

    def prolong(self, l, x):
        return torch.matmul(self.P[l], x.repeat_interleave(self.agg, 0).repeat_interleave(self.agg, 1))

    def vcycle(self, l, b):
        if l == len(self.P):
            return torch.matmul(self.inv, b.reshape(self.inv.shape[0], -1)).reshape(b.shape)
        D, x = self.D[l], torch.zeros_like(b)
        for _ in range(self.pre):
            x = D.sweep(b, x)
        x = x + self.prolong(l, self.vcycle(l + 1, self.restrict(l, b - D(x))))
        for _ in range(self.pre):
            x = D.sweep(b, x)
        return x

    def solve(self, l, b):
        """D_l x = b by restarted GCR with the V-cycle, every column to a true residual of 1e-13 or as far as it goes."""
        if l == len(self.P):
            return self.vcycle(l, b)
        D, x, goal = self.D[l], torch.zeros_like(b), 1e-13 * torch.linalg.vector_norm(b, dim=(0, 1, 2))
        for _ in range(12):
            r = b - D(x)
            if bool((torch.linalg.vector_norm(r, dim=(0, 1, 2)) <= goal).all()):
                break
            zs, ps = [], []
            for _ in range(10):
                z = self.vcycle(l, r)
                p = D(z)
                for z0, p0 in zip(zs, ps):
                    c = (p0.conj() * p).sum((0, 1, 2))
                    z, p = z - c * z0, p - c * p0
                nrm = torch.linalg.vector_norm(p, dim=(0, 1, 2)).clamp_min(1e-300)
                z, p = z / nrm, p / nrm
                c = (p.conj() * r).sum((0, 1, 2))
                x, r = x + c * z, r - c * p
                zs.append(z)
                ps.append(p)
        return x

    def difference(self, l, z):
        return self.solve(l, z) - self.prolong(l, self.solve(l + 1, self.restrict(l, z)))

    def noise(self, l, phase, seed, rhs, accumulated):
        """Noise vectors of level difference l, fine-size ones restricted to it in the accumulated form."""
        at = 0 if accumulated else l
        D = self.D[at]
        z = _signs(seed, l, phase, 0, rhs, D.L * D.L * D.d).to(C128)
        z = _to_field(z, D.L, D.d)
        for k in range(at, l):
            z = self.restrict(k, z)
        return z

    def sketch(self, l, d, k, seed, accumulated):
        s = self.noise(l, PHASE_SKETCH, seed, d, accumulated)
        for _ in range(k):
            y = self.difference(l, s)
            Q, R = torch.linalg.qr(y.reshape(-1, d))
            ph = R.diagonal()
            s = (Q * (ph / ph.abs())).reshape(y.shape)
        return s

    def project(self, Q, z, y):
        t = (z.conj() * y).sum((0, 1, 2))
        if Q is None:
            return t
        q, z, y = (v.reshape(-1, v.shape[-1]) for v in (Q, z, y))
        return t - ((q.mH @ z).conj() * (q.mH @ y)).sum(0)


def _to_field(x, L, d):
    return x.reshape(-1, L, L, d).permute(1, 2, 3, 0).contiguous()


def _to_rows(x):
    return x.permute(3, 0, 1, 2).reshape(x.shape[3], -1).contiguous()


def _exact_net(case, seed, U):
    """The network on bfloat16-rounded weights, every other number in 64 bits."""
    L, rhs = case["L"], case["rhs"]

    def sh(a, dx, dt):
        return a.roll((-dt, -dx), (0, 1))
    U0, U1 = U[..., 0], U[..., 1].clone()
    U1[L - 1] *= -1
    one = torch.ones_like(U0)
    Tx = {0: one, 1: U0, -1: sh(U0, -1, 0).conj()}
    Tt = {0: one, 1: U1, -1: sh(U1, 0, -1).conj()}
    W, b = _net_params(case["channels"], seed)
    par = []
    for l, w in enumerate(W):
        w = torch.from_numpy(np.stack([w.real, w.imag], -1).astype(np.float32)).to(torch.bfloat16)
        par.append(w.to(DEV, torch.float64).requires_grad_(case["grad"]))
        if l < len(b):
            par.append(torch.from_numpy(b[l].astype(np.float32)).to(DEV, torch.float64).requires_grad_(case["grad"]))
    r = _vectors(seed, rhs, 2 * L * L, C64).to(C128).reshape(rhs, L, L, 2)
    e = _vectors(seed, rhs, 2 * L * L, C64, 3).to(C128).reshape(rhs, L, L, 2)
    total, rows, per = 0.0, [], max(1, 2 ** 21 // (L * L * case["channels"]))
    for r0 in range(0, rhs, per):
        a, want = r[r0:r0 + per], e[r0:r0 + per]
        for l in range(len(W)):
            w, z = torch.view_as_complex(par[2 * l]), 0
            for d in range(9):
                dx, dt = d % 3 - 1, d // 3 - 1
                T = Tx[dx] * sh(Tt[dt], dx, 0)
                if dx and dt:
                    T = 0.5 * (T + Tt[dt] * sh(Tx[dx], 0, dt))
                z = z + torch.matmul(T[None, :, :, None] * a.roll((-dt, -dx), (1, 2)), w[d].T)
            if l + 1 < len(W):
                mag = z.abs()
                z = z * ((mag + par[2 * l + 1]).clamp_min(0) / mag)
            a = z
        if not case["grad"]:
            rows.append(a.reshape(len(a), -1))
            continue
        part = ((a - want).abs().square().sum((1, 2, 3)) / want.abs().square().sum((1, 2, 3))).sum() / rhs
        part.backward()
        total += float(part)
    if not case["grad"]:
        return torch.cat(rows)
    return total, torch.cat([p.grad.reshape(-1) for p in par]).cpu().numpy()


def exact(case, seed):
    op, L = case["op"], case["L"]
    U = _links(L, case["beta"], seed)
    n = 2 * L * L
    if op == "net":
        return _exact_net(case, seed, U)
    if op == "stencil":
        x = _vectors(seed, case["rhs"], n, C64 if case["prec"] == "fp32" else C128)
        D = _fine(U, case["m0"])
        return torch.cat([_to_rows(D(_to_field(p.to(C128), L, 2))) for p in x.split(max(1, 2 ** 24 // n))])
    if op == "hutchinson":
        D = _fine(U, case["m0"])
        z = _signs(seed, 0, PHASE_HUTCH, 0, case["samples"], n).to(C128).T
        M = D(torch.eye(n, dtype=C128, device=DEV).reshape(L, L, 2, n)).reshape(n, n)
        t = (z.conj() * torch.linalg.solve(M, z)).sum(0).cpu().numpy()
        return t.mean(), float(np.sqrt(np.var(t, ddof=1) / len(t))), t
    mg = _Multigrid(U, case["m0"], case.get("ntv", 8), case["sweeps"])
    if op == "vcycle":
        b = _vectors(seed, case["rhs"], n, C64 if case["prec"] == "fp32" else C128).to(C128)
        return _to_rows(mg.vcycle(0, _to_field(b, L, 2)))
    if op == "solve":
        z = _signs(seed, 0, PHASE_HUTCH, 0, case["rhs"], n).to(C128)
        return torch.cat([_to_rows(mg.solve(0, _to_field(p, L, 2))) for p in z.split(32)])
    if op == "setup":
        b = _vectors(seed, case["rhs"], n, C128)
        x = _to_rows(mg.vcycle(0, _to_field(b, L, 2)))
        return np.complex128(complex(mg.inv.trace())), x, x
    if op == "sample":
        l = min(case["level"], len(mg.P) - 1)
        z = mg.noise(l, PHASE_STOCH, seed, case["rhs"], False)
        y = mg.difference(l, z)
        Q = mg.sketch(l, case["d"], 1, seed, False) if case["d"] else None
        return mg.project(Q, z, y).cpu().numpy(), _to_rows(y)
    tau_L = complex(mg.inv.trace())
    lr, ts = [], []
    for l in range(len(mg.P)):
        Q = mg.sketch(l, case["d"], case["k"], seed, True)
        lr.append(complex((Q.conj() * mg.difference(l, Q)).sum()))
        z = mg.noise(l, PHASE_STOCH, seed, case["samples"], True)
        ts.append(mg.project(Q, z, mg.difference(l, z)).cpu().numpy())
    sigma = math.sqrt(sum(np.var(t, ddof=1) / len(t) for t in ts))
    return (np.complex128(sum(t.mean() for t in ts) + sum(lr) + tau_L), sigma, np.complex128(tau_L), np.array(lr),
            np.stack(ts))
