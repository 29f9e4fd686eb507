"""The kernels at the sizes where their work is split: molecules elongated along each axis and sizes
around the cell-list build's kernel choices, cells around 32 and 64 vertex slots (the clipping loop holds
one vertex per lane, and finishes larger cells elsewhere), Shrake-Rupley counts around the sizes of a
pass and of the neighbour groups, reused lists with pairs at tangency, and the limit on cells.

Tolerances are those of the parity tests; Shrake-Rupley counts follow stated float32 operations and
have to be equal."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
P = 1.4


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.fixture(scope="module")
def api():
    from paper_2401_10462_gb300 import api
    return api


def _run(api, torch, xyz, r, precision="mixed", ctx=None):
    own = ctx is None
    ctx = ctx or api.Context(precision=precision)
    n = len(r)
    a = torch.empty(n, dtype=torch.float64, device="cuda")
    g = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    ctx.compute(torch.as_tensor(np.ascontiguousarray(xyz), device="cuda"), torch.as_tensor(r, device="cuda"), a, g)
    ctx.status_sync()
    if own:
        ctx.close()
    return a.cpu().numpy(), g.cpu().numpy()


def _check(a, g, ra, rg):
    assert np.all(np.abs(a - ra) <= 1e-4 * np.maximum(ra, 1.0))
    assert abs(a.sum() - ra.sum()) <= 1e-6 * ra.sum()
    # 1e-3 relative, and the mixed form's rounding floor of 3e-5 where |g| < 0.03
    err = np.linalg.norm(g - rg, axis=1)
    assert np.all(err <= np.maximum(1e-3 * np.linalg.norm(rg, axis=1), 3e-5))


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n,seed", [(2047, 1), (2049, 2), (3040, 4), (3041, 5), (5001, 3)])
def test_elongated_along_each_axis(api, torch_cuda, orc, gen, axis, n, seed):
    """A long molecule along x (long runs of cells), y and z (many rows), on both sides of the one-block
    build's size and of the fused kernel's, far from the origin."""
    m = gen.rna(n, seed)
    x = np.roll(m.coords, axis - 2, axis=1) + np.array([300.0, -200.0, 100.0])
    a, g = _run(api, torch_cuda, x, m.radii)
    ra, _, rg = orc.sasa(x, m.radii)
    _check(a, g, ra, rg)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("m", [10, 17, 18, 19, 26, 33, 34])
def test_cells_around_the_slots_of_a_lane(api, torch_cuda, orc, m, precision):
    """A ball inside a shell of m small ones: its cell ends with 2 m - 4 vertices (16 .. 64), around 32
    slots (one per lane) and 64 (the fast pass)."""
    rng = np.random.default_rng(m)
    idx = np.arange(m) + 0.5
    z = 1 - 2 * idx / m
    rr = np.sqrt(1 - z * z)
    ang = math.pi * (1 + 5 ** 0.5) * idx
    shell = 5.2 * np.stack([rr * np.cos(ang), rr * np.sin(ang), z], 1) + 1e-4 * rng.normal(size=(m, 3))
    x = np.concatenate([np.full((1, 3), 1e-6), shell])
    r = np.concatenate([[3.6], np.full(m, 1.2)])
    a, g = _run(api, torch_cuda, x, r, precision)
    ra, _, rg = orc.sasa(x, r)
    _check(a, g, ra, rg)
    ctx = api.Context(precision=precision)
    torch = torch_cuda
    rec = ctx.export_complex(torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda")).cpu().numpy()
    ctx.close()
    o = orc.Oracle(x, r)
    for d in range(4):
        got = {tuple(int(v) for v in row[1:] if v >= 0) for row in rec if (row[1:] >= 0).sum() == d + 1}
        assert got == {tuple(int(v) for v in np.atleast_1d(s)) for s in o.simplices(d)}


def _sr_counts(x, r, pts):
    """The exposed counts by the stated float32 operations (no contraction)."""
    f = np.float32
    R = r + P
    out = []
    for i in range(len(r)):
        d = x - x[i]
        dd = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        rs = R + R[i]
        nb = np.nonzero(dd < rs * rs)[0]
        nb = nb[nb != i]
        p = f(R[i]) * pts
        free = np.ones(len(pts), bool)
        for j in nb:
            q = d[j].astype(f)
            e = p - q
            Rj = f(R[j])
            free &= ~((e[:, 0] * e[:, 0] + e[:, 1] * e[:, 1]) + e[:, 2] * e[:, 2] <= Rj * Rj)
        out.append(int(free.sum()))
    return np.array(out)


@pytest.mark.parametrize("m", [1, 31, 127, 128, 129, 257, 960])
@pytest.mark.parametrize("scale", [3.0, 1.6, 1.0, 0.72])
def test_shrake_rupley_counts(api, torch_cuda, gen, m, scale):
    """From isolated atoms (no neighbour) over a few (one group) to over sixty, with point numbers
    around one pass of 128."""
    torch = torch_cuda
    mol = gen.globule(120, 5)
    x, r = mol.coords * scale, mol.radii
    pts = gen.sphere_points(m)
    a = torch.empty(len(r), dtype=torch.float64, device="cuda")
    e = torch.empty(len(r), dtype=torch.int32, device="cuda")
    ctx = api.Context()
    ctx.compute_sr(torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda"),
                   torch.as_tensor(pts, device="cuda"), a, e)
    ctx.status_sync()
    ctx.close()
    ref = _sr_counts(x, r, pts)
    assert np.array_equal(e.cpu().numpy(), ref)
    assert np.allclose(a.cpu().numpy(), 4 * math.pi * (r + P) ** 2 * ref / m, rtol=1e-15)


@pytest.mark.parametrize("gap", [-1e-3, -1e-6, -1e-9, 0.0, 1e-9, 1e-6, 1e-3])
def test_reused_lists_at_tangency(api, torch_cuda, gap):
    """Pairs whose balls overlap by -gap, on a call that reuses its lists (float decides outside its
    rounding, float64 within it), against a context without lists."""
    rng = np.random.default_rng(7)
    n = 64
    r = rng.choice([1.2, 1.52, 1.7], size=2 * n)
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    centres = 40.0 * np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    d = (r[:n] + P) + (r[n:] + P) + gap
    x = np.concatenate([centres, centres + u * d[:, None]])
    ctx, plain = api.Context(skin=1.0), api.Context()
    _run(api, torch_cuda, x + 0.05 * rng.normal(size=x.shape), r, ctx=ctx)
    a, g = _run(api, torch_cuda, x, r, ctx=ctx)
    assert ctx.lists_reused()
    ra, rg = _run(api, torch_cuda, x, r, ctx=plain)
    assert np.allclose(a, ra, rtol=1e-6, atol=1e-6) and np.allclose(g, rg, rtol=1e-5, atol=3e-5)
    ctx.close()
    plain.close()


def _cubic_cells(x, r):
    """The cells of edge 2 R_max + slack in the molecule's box (what max_cells bounds)."""
    f = np.float32
    y = x.astype(f)
    lo, hi = y.min(0), y.max(0)
    amax = np.abs(np.concatenate([lo, hi])).max()
    margin = f(1e-5) + f(4e-7) * (amax + f(16))
    edge = f(2) * (r + P).astype(f).max() + f(2) * margin + f(1e-3)
    return int(np.prod(((hi - lo) / edge).astype(int) + 1))


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("sizes", [(300,), (3000,), (17000,), (300, 1500, 40, 700)])
def test_cell_limit(api, torch_cuda, orc, gen, sizes, axis):
    """max_cells: as many cubic cells as the molecules take are enough, one less is refused, and the
    context serves a molecule that fits afterwards."""
    torch = torch_cuda
    mols = [gen.rna(n, k) for k, n in enumerate(sizes)]
    x = [np.roll(m.coords, axis - 2, axis=1) for m in mols]
    cubes = sum(_cubic_cells(c, m.radii) for c, m in zip(x, mols))
    assert cubes > 64
    off = np.cumsum([0] + list(sizes))
    xs = torch.as_tensor(np.ascontiguousarray(np.concatenate(x)), device="cuda")
    rs = torch.as_tensor(np.concatenate([m.radii for m in mols]), device="cuda")
    for limit in (cubes, cubes - 1):
        ctx = api.Context(max_cells=limit)
        a = torch.empty(sum(sizes), dtype=torch.float64, device="cuda")
        if len(sizes) == 1:
            ctx.compute(xs, rs, a)
        else:
            ctx.compute_batch(off, xs, rs, a)
        if limit < cubes:
            assert ctx.status_code() == 3
            one = torch.empty(1, dtype=torch.float64, device="cuda")
            ctx.compute(torch.zeros((1, 3), dtype=torch.float64, device="cuda"),
                        torch.full((1,), 1.7, dtype=torch.float64, device="cuda"), one)
            ctx.status_sync()
            assert abs(one.item() - 4 * math.pi * 3.1 ** 2) <= 1e-9 * one.item()
        else:
            ctx.status_sync()
            ref = np.concatenate([orc.sasa(c, m.radii)[0] for c, m in zip(x, mols)])
            assert np.all(np.abs(a.cpu().numpy() - ref) <= 1e-4 * np.maximum(ref, 1.0))
        ctx.close()
