"""Cells that end in a rare way: emptied by a test that the filter leaves open, or emptied after one."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
P = 1.4


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("eps", [-1e-6, -1e-8, -1e-15, 0.0, 1e-15, 1e-8, 1e-6])
def test_emptied_at_a_corner(orc, eps, precision):
    """The deepest plane passes through the last corner of the initial cube, which is half-width
    h >= 1.0625 R + 0.0625 with a few bits, within eps: it leaves that corner or nothing, and a second
    plane takes the corner.  The ball's area is zero; all areas equal the oracle's within the mixed
    form's bounds."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import api
    R, d = 1.7 + P, 2.0
    h = math.ceil((R * 1.0625 + 0.0625) * 2 ** 20) / 2 ** 20
    big = math.sqrt(d * d + R * R + 2 * math.sqrt(3) * d * h) * (1 + eps)
    u, v = np.array([1.0, 1.0, 1.0]) / math.sqrt(3), np.array([1.0, 1.0, -1.0]) / math.sqrt(3)
    x = np.array([np.zeros(3), -d * u, -d * v, [9.0, 9.0, 9.0]])
    r = np.array([1.7, big - P, 0.999 * big - P, 1.5])
    xs, rs = torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda")
    a, g = torch.empty_like(rs), torch.empty_like(xs)
    ctx = api.Context(precision=precision)
    ctx.compute(xs, rs, a, g)
    ctx.status_sync()
    ctx.close()
    a, g = a.cpu().numpy(), g.cpu().numpy()
    ra, _, rg = orc.sasa(x, r)
    assert ra[0] == 0.0 and a[0] == 0.0 and np.all(g[0] == 0.0)
    assert np.all(np.abs(a - ra) <= 1e-4 * np.maximum(ra, 1.0))
    assert np.all(np.linalg.norm(g - rg, axis=1) <= np.maximum(1e-3 * np.linalg.norm(rg, axis=1), 3e-5))
