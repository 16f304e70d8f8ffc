"""Batches that do not fill a kernel's tile of right-hand sides cost in proportion to what they hold, and each
right-hand side's result does not depend on the batch it comes in."""
import numpy as np
import pytest

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
    for h in _HIER.values():
        h.close()
    _HIER.clear()
    c.close()


_HIER = {}


def hierarchy(api, ctx, L, **kw):
    key = (L, tuple(sorted(kw.items())))
    if key not in _HIER:
        U = np.exp(1j * np.random.default_rng(L).uniform(-0.9, 0.9, (L, L, 2)))
        par = dict(ntv=8, setup_sweeps=1, seed=3, tensor_cores=0)
        par.update(kw)
        _HIER[key] = api.mg_setup(ctx, torch.from_numpy(U).cuda(), L, 0.1, **par)
    return _HIER[key]


def vecs(n, k, seed, dtype):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((k, n), generator=g, dtype=dtype, device="cuda")


def micros(fn, reps=20, best=5):
    """Device time of one call among others, the best of a few series."""
    fn()
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    out = []
    for _ in range(best):
        torch.cuda.synchronize()
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b) / reps * 1e3)
    return min(out)


# level, lattice side, hierarchy, batch, larger batch, largest ratio of their times: FP64 units bound both, so the times
# go as the batches do (1/8, 9/16 and 17/32)
SMOOTH = [(0, 256, {}, 1, 8, 0.6), (0, 256, {}, 9, 16, 0.8), (0, 256, {}, 17, 32, 0.8),
          (1, 256, {}, 1, 8, 0.6), (1, 256, {}, 9, 16, 0.8), (1, 256, dict(ntv=4), 17, 32, 0.8)]


@pytest.mark.parametrize("level,L,kw,few,many,ratio", SMOOTH)
def test_smoother_cost(api, ctx, level, L, kw, few, many, ratio):
    """One FP64 sweep of `few` right-hand sides against one of `many`."""
    h = hierarchy(api, ctx, L, **kw)
    f, x = (vecs(h.n[level], many, s, torch.complex128) for s in (1, 2))
    t = [micros(lambda: h.smooth(level, f[:k], x[:k], api.FP64, 1)) for k in (few, many)]
    assert t[0] < ratio * t[1], t


@pytest.mark.parametrize("L,nrhs", [(16, 2), (16, 5), (32, 18), (64, 40), (384, 7), (384, 33)])
def test_fine_smoother_by_rhs(api, ctx, L, nrhs):
    """FP64 sweeps: tiles of 2 to 16 right-hand sides, spread over CTAs or looped over by one (from 4096 blocks of a
    colour on), with remainders of a warp's groups of 4, 2 and 1: the bits of one right-hand side at a time."""
    h = hierarchy(api, ctx, L, ntv=1)
    f, x = (vecs(h.n[0], nrhs, s, torch.complex128) for s in (1, 2))
    ref = x.clone()
    h.smooth(0, f, x, api.FP64, 2)
    for k in range(nrhs):
        h.smooth(0, f[k:k + 1], ref[k:k + 1], api.FP64, 2)
    assert torch.equal(x, ref)


@pytest.mark.parametrize("ntv,nrhs", [(8, 2), (8, 3), (8, 7), (8, 13), (4, 5), (4, 18), (2, 11), (2, 37), (1, 70)])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_coarse_smoother_by_rhs(api, ctx, ntv, nrhs, prec):
    """Sweeps on level 1 with 2 x 2 blocks of 8 to 64 unknowns (one to sixteen groups of rows in a CTA): batches that
    leave its groups uneven give the bits of one right-hand side at a time, also through the V-cycle's zero start."""
    h = hierarchy(api, ctx, 64, ntv=ntv)
    pr, dt = getattr(api, prec), torch.complex64 if prec == "FP32" else torch.complex128
    f, x = (vecs(h.n[1], nrhs, s, dt) for s in (1, 2))
    ref = x.clone()
    h.smooth(1, f, x, pr, 2)
    for k in range(nrhs):
        h.smooth(1, f[k:k + 1], ref[k:k + 1], pr, 2)
    assert torch.equal(x, ref)


def test_stopped_right_hand_sides(api, ctx):
    """Solves in which some right-hand sides never start (zero) or stop early beside others, FP64 and mixed: every
    solution satisfies the residual, whatever slots of a tile are live."""
    h = hierarchy(api, ctx, 64)
    b = vecs(h.n[0], 21, 5, torch.complex128)
    b[[0, 3, 4, 17]] = 0
    x = torch.empty_like(b)
    for prec in (api.FP64, api.MIXED):
        api.fgmres_batched(ctx, h, 0, b, x, tol=1e-10, prec=prec)
        r = torch.empty_like(b)
        h.apply(0, x, r, api.FP64)
        norm = torch.linalg.vector_norm
        assert (norm(b - r, dim=1) <= 1.1e-10 * norm(b, dim=1)).all() and not x[[0, 3, 4, 17]].any()


@pytest.mark.parametrize("few,many,ratio", [(1, 8, 0.6), (9, 16, 0.85)])
def test_restriction_cost(api, ctx, few, many, ratio):
    """FP64 restriction of `few` vectors of 16 dof per site against one of `many`."""
    h = hierarchy(api, ctx, 512)
    f, c = (vecs(h.n[l], many, l, torch.complex128) for l in (1, 2))
    t = [micros(lambda: h.restrict(1, f[:k], c[:k], api.FP64)) for k in (few, many)]
    assert t[0] < ratio * t[1], t


@pytest.mark.parametrize("L,nrhs", [(64, 3), (64, 5), (64, 37), (128, 13), (128, 50)])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_restriction_by_rhs(api, ctx, L, nrhs, prec):
    """Restriction from level 1 in tiles of 4, 8 and 16 right-hand sides with their remainders: the bits of one
    right-hand side at a time."""
    h = hierarchy(api, ctx, L)
    pr, dt = getattr(api, prec), torch.complex64 if prec == "FP32" else torch.complex128
    f = vecs(h.n[1], nrhs, 1, dt)
    c, ref = (torch.full((nrhs, h.n[2]), float("nan"), dtype=dt, device="cuda") for _ in range(2))
    h.restrict(1, f, c, pr)
    for k in range(nrhs):
        h.restrict(1, f[k:k + 1], ref[k:k + 1], pr)
    assert torch.equal(c, ref)


@pytest.mark.parametrize("level,L,prec,few,many,ratio", [(0, 512, "FP32", 8, 32, 0.5), (1, 256, "FP64", 9, 16, 0.85)])
def test_prolongation_cost(api, ctx, level, L, prec, few, many, ratio):
    """Prolongation of `few` vectors against one of `many`: on the fine level bound by memory (8 right-hand sides move a
    third of the bytes of 32), from 16 dof per site by the FP64 units."""
    h = hierarchy(api, ctx, L)
    pr, dt = getattr(api, prec), torch.complex64 if prec == "FP32" else torch.complex128
    f, c = (vecs(h.n[l], many, l, dt) for l in (level, level + 1))
    t = [micros(lambda: h.prolong(level, c[:k], f[:k], pr)) for k in (few, many)]
    assert t[0] < ratio * t[1], t


@pytest.mark.parametrize("L,nrhs", [(64, 2), (64, 7), (64, 9), (64, 35), (128, 13), (128, 41)])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_prolongation_by_rhs(api, ctx, L, nrhs, prec):
    """Prolongation to levels 0 and 1 in tiles of 8 and 32 right-hand sides with their remainders: the bits of one
    right-hand side at a time."""
    h = hierarchy(api, ctx, L)
    pr, dt = getattr(api, prec), torch.complex64 if prec == "FP32" else torch.complex128
    for l in range(2):
        c = vecs(h.n[l + 1], nrhs, 1, dt)
        f, ref = (torch.full((nrhs, h.n[l]), float("nan"), dtype=dt, device="cuda") for _ in range(2))
        h.prolong(l, c, f, pr)
        for k in range(nrhs):
            h.prolong(l, c[k:k + 1], ref[k:k + 1], pr)
        assert torch.equal(f, ref)


def test_coarsest_apply_cost(api, ctx):
    """FP64 inverse of a coarsest level of 1024 unknowns, applied one call behind the other: 32 right-hand sides load
    the SMs evenly (at most twice as long as the 16 that give every SM two tiles), 64 at most twice as long again."""
    h = hierarchy(api, ctx, 128)
    top = h.levels - 1
    b, x = (vecs(h.n[top], 64, s, torch.complex128) for s in (1, 2))
    t = [micros(lambda: h.vcycle(top, b[:k], x[:k], api.FP64)) for k in (16, 32, 64)]
    assert h.n[top] == 1024 and t[1] < 2.2 * t[0] and t[2] < 2.2 * t[1], t


@pytest.mark.parametrize("nrhs", [3, 11, 20, 33])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_coarsest_apply_by_rhs(api, ctx, nrhs, prec):
    """Warps of a tile without a right-hand side skip their products: the bits of one right-hand side at a time."""
    h = hierarchy(api, ctx, 64)
    top, pr, dt = h.levels - 1, getattr(api, prec), torch.complex64 if prec == "FP32" else torch.complex128
    b = vecs(h.n[top], nrhs, 1, dt)
    x, ref = (torch.full_like(b, float("nan")) for _ in range(2))
    h.vcycle(top, b, x, pr)
    for k in range(nrhs):
        h.vcycle(top, b[k:k + 1], ref[k:k + 1], pr)
    assert torch.equal(x, ref)


@pytest.mark.parametrize("L,nrhs", [(24, 22222), (72, 12346), (136, 3460)])
def test_stencil_lanes(api, ctx, L, nrhs):
    """FP32 operator on sides that are no multiple of its blocks: memory bounds it, so a batch takes the time that as
    many sites take at L = 512, up to a tenth (with idle lanes 1.16 to 1.23 times as long)."""
    t = []
    for side, k in ((L, nrhs), (512, max(1, round(nrhs * L * L / 512 ** 2)))):
        U = torch.from_numpy(np.exp(1j * np.random.default_rng(0).uniform(-3, 3, (side, side, 2)))).cuda()
        x = vecs(2 * side * side, k, 1, torch.complex64)
        y = torch.empty_like(x)
        t.append(micros(lambda: api.schwinger_apply(ctx, U, side, 0.1, x, y, api.FP32)) / (k * side * side))
    assert t[0] < 1.1 * t[1], t


@pytest.mark.parametrize("L,nrhs,rpt", [(142, 63, 1), (136, 76, 1), (130, 161, 2), (200, 65, 2), (130, 323, 4),
                                        (256, 101, 4), (142, 63, 4), (48, 700, 2)])
def test_stencil_walk_forms(api, ctx, L, nrhs, rpt):
    """The walking form with 1, 2 and 4 right-hand sides per thread set in the table, sides that are no multiple of its
    128 columns or 8 slices, batches that leave a thread short, a setting that would leave the chip short of threads
    (taken as 1) and a side below its smallest: against the FP64 form of the same call (nine terms, a few roundings of
    6e-8 each), and which kernel ran."""
    U = torch.from_numpy(np.exp(1j * np.random.default_rng(L).uniform(-3, 3, (L, L, 2)))).cuda()
    x = vecs(2 * L * L, nrhs, 3, torch.complex64)
    y = torch.full_like(x, float("nan"))
    x64 = x.to(torch.complex128)
    ref = torch.empty_like(x64)
    api.schwinger_apply(ctx, U, L, 0.1, x64, ref, api.FP64)
    bucket = 8
    while bucket < min(nrhs, 256):
        bucket *= 2
    try:
        api.tune_set([dict(kind=0, side=L, bucket=bucket, format=0, variant=rpt)])
        ctx.timing(True, "k_wilson")
        api.schwinger_apply(ctx, U, L, 0.1, x, y, api.FP32)
        ran = " ".join(ctx.timing_report())
    finally:
        ctx.timing(False)
        api.tune_clear()
    eff = 0 if L < 64 else rpt if L * L * nrhs / 8 / rpt >= 1024 * torch.cuda.get_device_properties(0).multi_processor_count else 1
    assert ("k_wilson_walk" in ran) == (eff > 0), (ran, eff)
    assert (y - ref).abs().max() < 2e-6 * ref.abs().max()


@pytest.mark.parametrize("level,nrhs,tiled", [(2, 1, False), (2, 16, False), (2, 17, True), (1, 1, True), (1, 16, True)])
def test_coarse_operator_forms(api, ctx, level, nrhs, tiled):
    """FP32 operator with 16 dof per site: 8 x 8 sites with up to 16 right-hand sides take the kernel of 256 threads per
    site, 16 x 16 sites and larger batches the tiled one (80 products, a few roundings of 6e-8 each)."""
    h = hierarchy(api, ctx, 128 if level == 2 else 64)
    x = vecs(h.n[level], nrhs, 1, torch.complex64)
    y, ref = torch.empty_like(x), torch.empty_like(x, dtype=torch.complex128)
    h.apply(level, x.to(torch.complex128), ref, api.FP64)
    try:
        ctx.timing(True, "k_coarse_apply")
        h.apply(level, x, y, api.FP32)
        ran = " ".join(ctx.timing_report())
    finally:
        ctx.timing(False)
    assert ("k_coarse_apply16" in ran) == tiled, ran
    assert (y - ref).abs().max() < 2e-5 * ref.abs().max()


def test_projection_chunks(api, ctx):
    """A projected sample's sums run over the same chunks of its rows whatever the batch: its bits do not depend on the
    other samples (one chunk of all rows for long batches would change them)."""
    h = hierarchy(api, ctx, 64)
    sk, _ = api.hutchpp_sketch_qr(ctx, h, 0, 8, 1, 3, api.ACCUMULATED, tol=1e-6, prec=api.MIXED)
    z, y = (vecs(h.n[0], 3000, s, torch.complex128) for s in (1, 2))
    tau = api.hutchpp_project(ctx, sk, z, y)
    for k in (0, 1500, 2999):
        assert api.hutchpp_project(ctx, sk, z[k:k + 1], y[k:k + 1])[0] == tau[k]
    sk.close()


def test_kernel_names_in_the_report(api, ctx):
    """Every launch of FP32 and FP64 cycles, sweeps and solves is reported under its kernel's name."""
    h = hierarchy(api, ctx, 128)
    try:
        ctx.timing(True)
        for pr, dt in ((api.FP32, torch.complex64), (api.FP64, torch.complex128)):
            b, x = (vecs(h.n[0], 3, s, dt) for s in (1, 2))
            h.vcycle(0, b, x, pr)
            api.fgmres_batched(ctx, h, 0, b, x, precond=0, m=4, tol=1e-30, maxit=4, prec=pr,
                               raise_on_nonconvergence=False)
        names = list(ctx.timing_report())
    finally:
        ctx.timing(False)
    assert any("k_sap_coarse" in n for n in names) and all(n.lstrip("(").startswith("k_") for n in names), names
