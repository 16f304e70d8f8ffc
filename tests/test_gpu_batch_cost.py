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


# level, lattice side, hierarchy, batch, larger batch, most that their times may differ by: FP64 units bound both, so
# the times go as the batches do (0.125, 0.56 and 0.53 here)
SMOOTH = [(0, 256, {}, 1, 8, 0.6), (0, 256, {}, 9, 16, 0.8), (0, 256, {}, 17, 32, 0.8)]


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
