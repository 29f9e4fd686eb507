"""Long molecules, whose cell grid has long rows or reaches its limit of cells along an axis: pairs of
overlapping atoms far from one another, whose exposed areas and gradients have a closed form."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
P = 1.4


def _pairs(n, length, axis):
    """n atoms in n / 2 pairs along an axis, and their areas and gradients of the total area."""
    k = np.arange(n // 2)
    x = np.zeros((n, 3))
    x[0::2, axis] = (k / (n // 2 - 1) - 0.5) * length
    x[1::2, axis] = x[0::2, axis] + 2.5
    r = np.where(k % 2 == 0, 1.8, 1.5).repeat(2)
    R = r + P
    d = x[1::2, axis] - x[0::2, axis]
    # equal radii: each ball loses a cap of height R - d / 2
    area = 2 * math.pi * R * (R + d.repeat(2) / 2)
    grad = np.zeros((n, 3))
    grad[1::2, axis] = 2 * math.pi * R[1::2]
    grad[0::2, axis] = -2 * math.pi * R[0::2]
    return x, r, area, grad


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("axis,n,length", [(0, 130000, 1.9e6), (0, 260000, 2e7), (1, 300000, 2e7), (2, 300000, 2e7)])
def test_pairs_along_an_axis(axis, n, length, batch):
    """1.05 million cells would lie along x, and more than a million along y and z: an axis holds a
    million, and atoms past its end must keep their neighbours.  Bounds: the mixed form's (areas
    1e-4; gradients 1e-3 relative)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import api
    x, r, area, grad = _pairs(n, length, axis)
    off = [0, n]
    if batch:   # a small molecule before it
        x = np.concatenate([x[n // 2:n // 2 + 2], x])
        r, area, grad = (np.concatenate([v[n // 2:n // 2 + 2], v]) for v in (r, area, grad))
        off = [0, 2, n + 2]
    xs, rs = torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda")
    a, g = torch.empty_like(rs), torch.empty_like(xs)
    ctx = api.Context()
    if batch:
        ctx.compute_batch(np.array(off), xs, rs, a, g)
    else:
        ctx.compute(xs, rs, a, g)
    ctx.status_sync()
    ctx.close()
    assert np.all(np.abs(a.cpu().numpy() - area) <= 1e-4 * area)
    err = np.linalg.norm(g.cpu().numpy() - grad, axis=1)
    assert np.all(err <= 1e-3 * np.linalg.norm(grad, axis=1))


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import api
    return torch, api


def _lines(row, k):
    """3,296 atoms in pairs on k x k lines along x, 10 A apart, whose box is `row` cells long."""
    reach, length = 2 * (1.8 + P), 0.0
    for _ in range(4):   # a cell is a quarter of the edge, the edge the reach with its slack
        edge = reach + 2 * (1e-5 + 4e-7 * (length / 2 + 16)) + 1e-3
        length = (row - 0.5) * edge / 4
    x, r, area, grad = _pairs(3296 // (k * k), length - 2.5, 0)
    x[:, 0] -= 1.25
    off = 10.0 * np.stack(np.meshgrid([0], np.arange(k), np.arange(k), indexing="ij"), -1).reshape(-1, 1, 3)
    return ((x + off).reshape(-1, 3), np.tile(r, k * k), np.tile(area, k * k), np.tile(grad, (k * k, 1)))


@pytest.mark.parametrize("row,k", [(1023, 4), (1024, 4), (1025, 4), (4094, 2), (4095, 2), (4096, 2), (4900, 2)])
def test_row_lengths(env, row, k):
    """Rows of cells around the length from which whole blocks scan them, and around a block's tile of
    4096 cells.  Bounds as above."""
    torch, api = env
    x, r, area, grad = _lines(row, k)
    xs, rs = torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda")
    a, g = torch.empty_like(rs), torch.empty_like(xs)
    ctx = api.Context()
    for _ in range(2):
        ctx.compute(xs, rs, a, g)
    ctx.status_sync()
    ctx.close()
    assert np.all(np.abs(a.cpu().numpy() - area) <= 1e-4 * area)
    err = np.linalg.norm(g.cpu().numpy() - grad, axis=1)
    assert np.all(err <= 1e-3 * np.linalg.norm(grad, axis=1))


def test_a_fibre_takes_no_longer_along_x(env):
    """130,000 atoms in one row of a million cells, against the same ones in a million rows."""
    torch, api = env
    ms = []
    for axis in (0, 1):
        x, r, _, _ = _pairs(130000, 1.8e6, axis)
        xs, rs = torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda")
        a, g = torch.empty_like(rs), torch.empty_like(xs)
        ctx = api.Context()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(8)]
        for e in ev:
            e.record()
            ctx.compute(xs, rs, a, g)
        ctx.status_sync()
        ctx.close()
        ms.append(min(ev[k].elapsed_time(ev[k + 1]) for k in range(3, 7)))
    assert ms[0] <= 2.0 * ms[1], ms
