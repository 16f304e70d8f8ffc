"""Kernels at the edges of their tiles (remainders of the right-hand-side and row tiles, smallest lattices), against
the CPU oracle.  Tolerances are relative to the largest reference entry and stated from the arithmetic: FP64 kernels
a few hundred roundings of 1.1e-16 (1e-12 where block inverses enter), FP32 ones of 6e-8."""
import numpy as np
import pytest

from oracle import multigrid as omg
from oracle import schwinger as osch
from synthetic import gauge

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2303_11512_gb300 import api
    return api


@pytest.fixture(scope="module")
def ctx(api):
    c = api.Context()
    yield c
    for h, _ in _HIER.values():
        h.close()
    _HIER.clear()
    c.close()


_HIER = {}


def hierarchy(api, ctx, L, **kw):
    """(GPU hierarchy, oracle hierarchy) of one interacting field without bootstrap rounds."""
    key = (L, tuple(sorted(kw.items())))
    if key not in _HIER:
        U = gauge.links(gauge.field(L, 3.0, 0, sweeps=60))
        par = dict(ntv=4, setup_sweeps=2, seed=3, tensor_cores=0, pre_smooth=1, post_smooth=1)
        par.update(kw)
        h = api.mg_setup(ctx, torch.from_numpy(U).cuda(), L, -0.05, **par)
        H = omg.Hierarchy(osch.dirac_sparse(U, -0.05), L, ntv=par["ntv"], setup_sweeps=2, seed=3)
        _HIER[key] = (h, H)
    return _HIER[key]


def relerr(a, b):
    return float(np.abs(np.asarray(a) - b).max() / np.abs(b).max())


def vecs(n, k, seed, dtype):
    rs = np.random.default_rng(seed)
    return (rs.standard_normal((k, n)) + 1j * rs.standard_normal((k, n))).astype(dtype)


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-12), ("FP32", 2e-5)])
@pytest.mark.parametrize("L,nrhs", [(16, 1), (16, 8), (16, 9), (16, 17), (32, 33)])
def test_fine_smoother_and_cycle_tiles(api, ctx, L, nrhs, prec, tol):
    """Fine SAP sweeps from a given x and, through the V-cycle, from zero: rhs tiles of 8 and 16 and their remainders
    (one 4 x 4 block solve amplifies roundings by its condition, about 10, over at most 4 half sweeps)."""
    h, H = hierarchy(api, ctx, L)
    dt = np.complex128 if prec == "FP64" else np.complex64
    f, x = vecs(H.n[0], nrhs, 1, dt), vecs(H.n[0], nrhs, 2, dt)
    ref = H.sap(0).sweep(f.T.astype(complex), x.T.astype(complex)).T
    xd = torch.from_numpy(x).cuda()
    h.smooth(0, torch.from_numpy(f).cuda(), xd, getattr(api, prec), 1)
    assert relerr(xd.cpu().numpy(), ref) < tol
    xd.fill_(float("nan"))  # the cycle starts from zero whatever the output buffer holds
    h.vcycle(0, torch.from_numpy(f).cuda(), xd, getattr(api, prec))
    assert relerr(xd.cpu().numpy(), H.vcycle(0, f.T, 1, 1).T) < 10 * tol


@pytest.mark.parametrize("L,nrhs,m", [(16, 1, 1), (16, 5, 30), (32, 33, 40), (64, 3, 16), (80, 2, 24), (128, 2, 20)])
@pytest.mark.parametrize("prec", ["FP64", "FP32"])
def test_krylov_step_forms(api, ctx, L, nrhs, m, prec):
    """GMRES without preconditioner in the one-launch form (up to 16384 entries: 512, 2048, 8192, 12800) and the
    three-pass form (32768), past 16 basis vectors, at restart lengths 1 and 40: the true residual, computed by the
    oracle's operator, is what the solver promises (FP32: its own rounding, 6e-8 of a residual amplified by the 6
    terms of a row, allows 1e-5)."""
    U = gauge.links(gauge.field(L, 3.0, 0, sweeps=10))
    m0 = 0.2  # well conditioned: the point is the arithmetic of a step
    h = api.mg_setup(ctx, torch.from_numpy(U).cuda(), L, m0, ntv=1, setup_sweeps=1, tensor_cores=0, levels=2)
    try:
        D = osch.dirac_sparse(U, m0)
        dt, tol = (np.complex128, 1e-10) if prec == "FP64" else (np.complex64, 1e-5)
        b = vecs(2 * L * L, nrhs, 4, dt)
        b[0] *= 1e6  # per-rhs norms and stops
        bd = torch.from_numpy(b).cuda()
        xd = torch.empty_like(bd)
        st = api.fgmres_batched(ctx, h, 0, bd, xd, precond=0, m=m, tol=tol, prec=getattr(api, prec), maxit=4000)
        x = xd.cpu().numpy().astype(complex)
        res = np.linalg.norm(b - (D @ x.T).T, axis=1) / np.linalg.norm(b, axis=1)
        assert st["converged"] and res.max() < 1.5 * tol, res
        assert st["its"].min() > 0
    finally:
        h.close()


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-12), ("FP32", 1e-5)])
@pytest.mark.parametrize("nrhs", [1, 8, 9, 17, 65])
def test_coarsest_apply_tiles(api, ctx, nrhs, prec, tol):
    """The coarsest level's dense inverse at the remainders of its 8 and 16 rhs tiles (sums of 128 products; the
    inverse's condition, below 100, is in the tolerance)."""
    h, H = hierarchy(api, ctx, 16)
    top = h.levels - 1
    b = vecs(H.n[top], nrhs, 6, np.complex128 if prec == "FP64" else np.complex64)
    xd = torch.empty(b.shape, dtype=torch.from_numpy(b).dtype, device="cuda")
    h.vcycle(top, torch.from_numpy(b).cuda(), xd, getattr(api, prec))
    assert relerr(xd.cpu().numpy(), H.vcycle(top, b.T).T) < tol


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-12), ("FP32", 2e-5)])
@pytest.mark.parametrize("ntv,nrhs", [(4, 1), (4, 17), (8, 8), (8, 9), (1, 33)])
def test_coarse_smoother_tiles(api, ctx, ntv, nrhs, prec, tol):
    """SAP sweeps on level 1 on the CUDA cores (2 x 2 blocks of 2, 8 and 16 dof per site), remainders of the rhs tile
    (tolerances as for the fine smoother: block condition about 10)."""
    h, H = hierarchy(api, ctx, 64, ntv=ntv)
    dt = np.complex128 if prec == "FP64" else np.complex64
    f, x = vecs(H.n[1], nrhs, 1, dt), vecs(H.n[1], nrhs, 2, dt)
    ref = H.sap(1).sweep(f.T.astype(complex), x.T.astype(complex)).T
    xd = torch.from_numpy(x).cuda()
    h.smooth(1, torch.from_numpy(f).cuda(), xd, getattr(api, prec), 1)
    assert relerr(xd.cpu().numpy(), ref) < tol


@pytest.mark.parametrize("n", [33, 40, 250, 257, 600])
@pytest.mark.parametrize("prec,eps", [("FP64", 1.1e-16), ("FP32", 6e-8)])
def test_dense_inverse_block_columns(api, ctx, n, prec, eps):
    """Remainders of the 8-column blocks, of the cluster's row shares and of the 32 x 32 update tiles, with a zero
    leading entry so that rows are swapped from the first column on: A times the inverse is the identity to n
    roundings amplified by the condition number."""
    rs = np.random.default_rng(n)
    A = (rs.standard_normal((n, n)) + 1j * rs.standard_normal((n, n))).astype(
        np.complex128 if prec == "FP64" else np.complex64)
    A[0, 0] = 0
    B = torch.from_numpy(A).cuda()
    api.mg_dense_inverse(ctx, B, getattr(api, prec))
    A = A.astype(complex)
    err = np.abs(B.cpu().numpy() @ A - np.eye(n)).max()
    assert err < n * eps * np.linalg.cond(A)
    S = torch.zeros((n, n), dtype=B.dtype, device="cuda")
    S[0, 1] = S[1, 0] = 1  # singular from the third column on
    with pytest.raises(Exception):
        api.mg_dense_inverse(ctx, S, getattr(api, prec))


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-13), ("FP32", 5e-6)])
@pytest.mark.parametrize("nrhs", [1, 8, 9, 33])
@pytest.mark.parametrize("shift", [0, 1])
def test_transfer_tiles(api, ctx, nrhs, prec, tol, shift):
    """Restriction and prolongation of both levels (2 and 16 dof) at the remainders of the rhs tiles, and on vectors
    that start 8 bytes off a 16-byte boundary in FP32 (up to 256 products, roundings of order eps each)."""
    h, H = hierarchy(api, ctx, 64, ntv=8)
    dt = np.complex128 if prec == "FP64" else np.complex64
    for l in range(2):
        xf, xc = vecs(H.n[l], nrhs, 1, dt), vecs(H.n[l + 1], nrhs, 2, dt)
        def off(a):
            buf = torch.empty(a.size + shift, dtype=torch.from_numpy(a).dtype, device="cuda")
            v = buf[shift:].view(a.shape)
            v.copy_(torch.from_numpy(a))
            return v
        f, c = off(xf), off(np.zeros_like(xc))
        h.restrict(l, f, c, getattr(api, prec))
        assert relerr(c.cpu().numpy(), (H.P[l].conj().T @ xf.T.astype(complex)).T) < tol
        h.prolong(l, off(xc), f, getattr(api, prec))
        assert relerr(f.cpu().numpy(), (H.P[l] @ xc.T.astype(complex)).T) < tol


@pytest.mark.parametrize("images,tol", [(0, 2e-4), (1, 5e-2), (2, 1e-2), (3, 1e-2)])
@pytest.mark.parametrize("nrhs", [1, 17, 40])
def test_cycle_with_fused_transfers(api, ctx, nrhs, images, tol):
    """Three-level FP32 V-cycle: fused residual and restriction on the fine level, the half restriction after a
    tensor-core sweep (16-bit formats round at 4e-3 / 5e-4, TF32 at 5e-4, several times along a cycle)."""
    h, H = hierarchy(api, ctx, 64, ntv=8, tensor_cores=images)
    b = vecs(H.n[0], nrhs, 5, np.complex64)
    xd = torch.full(b.shape, float("nan"), dtype=torch.complex64, device="cuda")
    h.vcycle(0, torch.from_numpy(b).cuda(), xd, api.FP32)
    assert relerr(xd.cpu().numpy(), H.vcycle(0, b.T.astype(complex), 1, 1).T) < tol


@pytest.mark.parametrize("L,nrhs", [(4, 1), (6, 7), (130, 80), (142, 61), (512, 5), (512, 6)])
@pytest.mark.parametrize("prec,tol", [("FP64", 1e-14), ("FP32", 2e-6)])
def test_stencil_forms(api, ctx, L, nrhs, prec, tol):
    """Fine operator straight from U (up to 64 K sites x rhs), from prepared links, and walking along t with lattice
    sides that are no multiple of its 128 columns or 8 slices (nine terms, a few roundings each)."""
    rs = np.random.default_rng(L)
    U = np.exp(1j * rs.uniform(-3, 3, (L, L, 2)))
    dt = np.complex128 if prec == "FP64" else np.complex64
    x = vecs(2 * L * L, nrhs, 3, dt)
    y = torch.full(x.shape, float("nan"), dtype=torch.from_numpy(x).dtype, device="cuda")
    api.schwinger_apply(ctx, torch.from_numpy(U).cuda(), L, 0.1, torch.from_numpy(x).cuda(), y, getattr(api, prec))
    ref = (osch.dirac_sparse(U, 0.1) @ x.T.astype(complex)).T
    assert relerr(y.cpu().numpy(), ref) < tol


@pytest.mark.parametrize("nrhs", [1, 16, 17, 33])
@pytest.mark.parametrize("shift", [0, 1])
def test_coarse_operator_tiles(api, ctx, nrhs, shift):
    """FP32 operator with 16 dof per site at the remainders of its rhs tiles, also on vectors that start 8 bytes off
    a 16-byte boundary (80 products, a few roundings of 6e-8 each)."""
    h, H = hierarchy(api, ctx, 64, ntv=8)
    x = vecs(H.n[1], nrhs, 7, np.complex64)
    buf = torch.empty(x.size + shift, dtype=torch.complex64, device="cuda")
    xd = buf[shift:].view(x.shape)
    xd.copy_(torch.from_numpy(x))
    y = torch.full(x.shape, float("nan"), dtype=torch.complex64, device="cuda")
    h.apply(1, xd, y, api.FP32)
    assert relerr(y.cpu().numpy(), (H.D[1] @ x.T.astype(complex)).T) < 2e-5


@pytest.mark.parametrize("d,nrhs", [(1, 1), (7, 9), (8, 17), (9, 5), (24, 24), (33, 8), (64, 33)])
def test_projection_tiles(api, ctx, d, nrhs):
    """Projected samples at the remainders of the basis and rhs tiles (sums of 512 products, their roundings)."""
    h, H = hierarchy(api, ctx, 16)
    sk, _ = api.hutchpp_sketch_qr(ctx, h, 0, d, 1, 3, api.ACCUMULATED, tol=1e-6, prec=api.MIXED)
    Q = sk.Q().cpu().numpy()
    z, y = vecs(H.n[0], nrhs, 1, np.complex128), vecs(H.n[0], nrhs, 2, np.complex128)
    tau = api.hutchpp_project(ctx, sk, torch.from_numpy(z).cuda(), torch.from_numpy(y).cuda())
    zp = z - (z @ Q.conj().T) @ Q
    assert relerr(tau, np.einsum("ij,ij->i", zp.conj(), y)) < 1e-12


@pytest.mark.parametrize("d", [1, 2, 31, 32, 33, 63])
def test_cholesky_qr_sizes(api, ctx, d):
    """Orthonormal basis by the Cholesky factor's right-looking form: Q^H Q = I to a few hundred roundings."""
    Y = torch.from_numpy(vecs(1000, d, d, np.complex128)).cuda()
    ref = Y.cpu().numpy()
    api.hutchpp_cholqr2(ctx, Y)
    Q = Y.cpu().numpy()
    R = Q.conj() @ ref.T  # Y = R^T Q by rows: upper triangular with a positive real diagonal
    assert np.abs(Q.conj() @ Q.T - np.eye(d)).max() < 1e-13
    assert np.abs(np.tril(R, -1)).max(initial=0) < 1e-11 and np.diag(R).real.min() > 0


def test_stencil_in_a_stream_capture(api):
    """The first call of a context inside a stream capture keeps nothing of the capture's memory: calls after it, and
    replays, give the same values as a call of another context."""
    L, nrhs = 128, 8
    U = torch.from_numpy(np.exp(1j * np.random.default_rng(0).uniform(-3, 3, (L, L, 2)))).cuda()
    x = torch.from_numpy(vecs(2 * L * L, nrhs, 3, np.complex128)).cuda()
    ref, y, z = (torch.zeros_like(x) for _ in range(3))
    c = api.Context()
    api.schwinger_apply(c, U, L, 0.1, x, ref, api.FP64)
    c.close()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    c = api.Context(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        api.schwinger_apply(c, U, L, 0.1, x, y, api.FP64)
    api.schwinger_apply(c, U, L, 0.1, x, z, api.FP64)
    with torch.cuda.stream(s):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(z, ref) and torch.equal(y, ref)
    c.close()


def test_batches_beyond_the_grid(api, ctx):
    """Operators, transfers and smoothers on more right-hand sides than one grid holds tiles of: the last ones equal a
    batch of their own (the same sums, up to a few roundings of 6e-8 in another tile shape)."""
    h, H = hierarchy(api, ctx, 16, ntv=8)
    nrhs, k = 16 * 65535 + 5, 7
    f = torch.zeros((nrhs, H.n[1]), dtype=torch.complex64, device="cuda")
    f[-k:] = torch.from_numpy(vecs(H.n[1], k, 1, np.complex64)).cuda()
    out, ref = torch.empty_like(f), torch.empty_like(f[-k:])
    h.apply(1, f, out, api.FP32)
    h.apply(1, f[-k:].clone(), ref, api.FP32)
    assert relerr(out[-k:].cpu().numpy(), ref.cpu().numpy()) < 2e-6
    del out
    fine = torch.zeros((nrhs, H.n[0]), dtype=torch.complex64, device="cuda")
    fref = torch.empty((k, H.n[0]), dtype=torch.complex64, device="cuda")
    h.prolong(0, f, fine, api.FP32)
    h.prolong(0, f[-k:].clone(), fref, api.FP32)
    assert relerr(fine[-k:].cpu().numpy(), fref.cpu().numpy()) < 2e-6
    h.restrict(0, fine, f, api.FP32)
    h.restrict(0, fref, ref, api.FP32)
    assert relerr(f[-k:].cpu().numpy(), ref.cpu().numpy()) < 2e-6
    x, xref = torch.zeros_like(fine), torch.zeros_like(fref)
    h.smooth(0, fine, x, api.FP32, 1)
    h.smooth(0, fref, xref, api.FP32, 1)
    assert relerr(x[-k:].cpu().numpy(), xref.cpu().numpy()) < 2e-6


@pytest.mark.parametrize("n", [1, 2, 7, 31, 32, 33])
@pytest.mark.parametrize("prec,eps", [("FP64", 1.1e-16), ("FP32", 6e-8)])
def test_dense_inverse_without_barrier(api, ctx, n, prec, eps):
    """Without a poll limit no size runs the kernel that spins on a grid barrier (n <= 32: one CTA, 33 on: block
    columns); the inverse of a matrix whose rows have to be swapped, against the identity as above, and a singular one."""
    rs = np.random.default_rng(n)
    A = (rs.standard_normal((n, n)) + 1j * rs.standard_normal((n, n))).astype(
        np.complex128 if prec == "FP64" else np.complex64)
    if n > 1:
        A[0, 0] = 0
    B = torch.from_numpy(A).cuda()
    try:
        ctx.timing(True)
        api.mg_dense_inverse(ctx, B, getattr(api, prec))
        ran = " ".join(ctx.timing_report())
    finally:
        ctx.timing(False)
    assert "k_gj_coop" not in ran and ("k_gj_panel" in ran) == (n > 32), ran
    A = A.astype(complex)
    assert np.abs(B.cpu().numpy() @ A - np.eye(n)).max() < 4 * n * eps * np.linalg.cond(A)
    with pytest.raises(Exception):
        api.mg_dense_inverse(ctx, torch.zeros((n, n), dtype=B.dtype, device="cuda"), getattr(api, prec))


def free_field(L, periodic=False):
    U = np.ones((L, L, 2), dtype=complex)
    if periodic:
        U[L - 1, :, 1] = -1  # undoes the antiperiodic sign
    return U


def test_reported_bytes_follow_the_stopped(api, ctx):
    """Unpreconditioned solve of seven plane waves of the free field, each done in two steps, beside a random vector of
    many: the report bills the operator for the right-hand sides that go on, at most two steps late."""
    L, nrhs = 32, 8
    U = free_field(L)
    h = api.mg_setup(ctx, torch.from_numpy(U).cuda(), L, 0.2, ntv=1, setup_sweeps=1, tensor_cores=0, levels=2)
    try:
        t, x = np.meshgrid(np.arange(L), np.arange(L), indexing="ij")
        b = vecs(2 * L * L, nrhs, 1, np.complex128)
        for k in range(nrhs - 1):
            wave = np.exp(2j * np.pi * ((k + 0.5) * t + 3 * k * x) / L)
            b[k] = (wave[..., None] * np.array([0.3, 0.7 + 0.2j])).reshape(-1)
        bd = torch.from_numpy(b).cuda()
        xd = torch.empty_like(bd)
        ctx.timing(True, "k_wilson")
        st = api.fgmres_batched(ctx, h, 0, bd, xd, precond=0, m=64, tol=1e-10, prec=api.FP64, maxit=60,
                                raise_on_nonconvergence=False)
        rep = ctx.timing_report()
        ctx.timing(False)
        steps = int(st["its"].max())
        assert steps >= 20 and sorted(st["its"])[-2] <= 3, st["its"]
        full = 32.0 * L * L * (2 * nrhs + 1)  # bytes of one application to the whole batch
        used = sum(r["bytes"] for r in rep.values()) / full
        assert used < 4 + 0.25 * steps, (used, steps)
    finally:
        ctx.timing(False)
        h.close()


@pytest.mark.parametrize("L", [16, 32, 64, 128])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_spent_krylov_space(api, ctx, L, prec):
    """An eigenvector (the constant spinor of the periodic free field) spends its Krylov space in one step, up to a
    residue of rounding that lies in the span: the cycle ends there, in the one-launch form (up to 16384 entries) and in
    the three-pass form, and the true residual decides.  Plane waves of two spin components spend it in two."""
    dt, eps = (np.complex64, 6e-8) if prec == "FP32" else (np.complex128, 1.1e-16)
    t, x = np.meshgrid(np.arange(L), np.arange(L), indexing="ij")
    for m0 in (0.2, 0.37, 0.61):
        for periodic in (True, False):
            U = free_field(L, periodic)
            h = api.mg_setup(ctx, torch.from_numpy(U).cuda(), L, m0, ntv=1, setup_sweeps=1, tensor_cores=0,
                             levels=2 if L <= 64 else 0)
            try:
                D = osch.dirac_sparse(U, m0)
                wave = np.ones((L, L)) if periodic else np.exp(2j * np.pi * (2.5 * t + 3 * x) / L)
                b = (wave[..., None] * np.array([1, 1] if periodic else [0.3, 0.7 + 0.2j])).reshape(1, -1).astype(dt)
                bd = torch.from_numpy(b).cuda()
                xd = torch.empty_like(bd)
                st = api.fgmres_batched(ctx, h, 0, bd, xd, precond=0, m=30, tol=1e-300, maxit=12, prec=getattr(api, prec),
                                        raise_on_nonconvergence=False)
                res = np.linalg.norm(b[0] - D @ xd.cpu().numpy()[0].astype(complex)) / np.linalg.norm(b)
                assert res < 100 * eps, res
                if periodic:
                    assert st["its"][0] == st["outer"], st
            finally:
                h.close()


def test_unpreconditioned_memory(api):
    """A solve without preconditioner holds one basis of m + 1 batches: 33 of 34 MB here, and 32 more with a second."""
    L, nrhs, m = 128, 64, 32
    c = api.Context()
    h = api.mg_setup(c, torch.from_numpy(free_field(L)).cuda(), L, 0.5, ntv=1, setup_sweeps=1, tensor_cores=0)
    try:
        b = torch.from_numpy(vecs(2 * L * L, nrhs, 1, np.complex128)).cuda()
        x = torch.empty_like(b)
        api.fgmres_batched(c, h, 0, b, x, precond=0, m=1, tol=0.9, prec=api.FP64)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        api.fgmres_batched(c, h, 0, b, x, precond=0, m=m, tol=1e-3, prec=api.FP64)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
        batch = 16 * 2 * L * L * nrhs
        assert used < 1.3 * (m + 1) * batch, used / batch
    finally:
        h.close()
        c.close()


@pytest.mark.parametrize("L,level,ntv,prec,tol", [(16, 0, 8, "FP32", 2e-5), (16, 0, 8, "FP64", 1e-12),
                                                  (64, 1, 8, "FP32", 2e-5), (64, 1, 4, "FP64", 1e-12)])
def test_cycles_beyond_one_slice(api, ctx, L, level, ntv, prec, tol):
    """V-cycles and sweeps of more right-hand sides than the tiled kernels take in one slice (256 K): smoothers of both
    levels, fused residual and restriction, operator, transfers and coarsest apply in both precisions; the last
    right-hand sides equal a batch of their own (the same sums, in FP32 up to roundings in another tile shape)."""
    h, H = hierarchy(api, ctx, L, ntv=ntv)
    pr, dt = getattr(api, prec), torch.complex64 if prec == "FP32" else torch.complex128
    nrhs, k = (1 << 18) + 5, 7
    f = torch.zeros((nrhs, H.n[level]), dtype=dt, device="cuda")
    f[-k:] = torch.from_numpy(vecs(H.n[level], k, 1, np.complex128)).cuda().to(dt)
    x = torch.zeros_like(f)
    ref = torch.zeros_like(f[-k:])
    for call in (lambda b, y: h.smooth(level, b, y, pr, 1), lambda b, y: h.vcycle(level, b, y, pr)):
        call(f, x)
        call(f[-k:].clone(), ref)
        assert relerr(x[-k:].cpu().numpy(), ref.cpu().numpy()) < tol and not x[:-k].any()
    del f, x
    torch.cuda.empty_cache()
