"""Molecules so long that the cell grid reaches its limit of cells along an axis: pairs of overlapping
atoms far from one another, whose exposed areas and gradients have a closed form."""
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
