"""The initial cube's half-width (csrc/dsasa_math.cuh, compiled for the host by g++): its planes have to
be the same numbers in float and in double, for every radius, since filters and exact predicates
decide about one cube; and cells of large balls on the GPU against the oracle."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
HDR = os.path.join(ROOT, "paper_2401_10462_gb300", "csrc", "dsasa_math.cuh")
SO = os.path.join(ROOT, "paper_2401_10462_gb300", "_build", "libghostcheck.so")
SRC = f'#include "{HDR}"\nextern "C" double gc_h(double r) {{ return dsasa::ghost_h(r); }}\n'
P = 1.4


@pytest.fixture(scope="module")
def half_width():
    os.makedirs(os.path.dirname(SO), exist_ok=True)
    tmp = SO + f".tmp{os.getpid()}"
    subprocess.run(["g++", "-x", "c++", "-", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-o", tmp],
                   input=SRC.encode(), check=True)
    os.replace(tmp, SO)
    f = ctypes.CDLL(SO).gc_h
    f.argtypes, f.restype = [ctypes.c_double], ctypes.c_double
    return f


def test_half_width_is_a_float(half_width):
    rng = np.random.default_rng(0)
    for R in np.concatenate([10.0 ** rng.uniform(-3, 9, 4000), [14.9, 15.0, 15.06, 16.0, 30.0, 31.0, 1e6]]):
        h = half_width(R)
        assert float(np.float32(h)) == h
        assert Fraction(2.0 * h) == 2 * Fraction(h) and Fraction(2.0 * h * h) == 2 * Fraction(h) ** 2
        assert R * 1.0625 < h <= (R * 1.0625 + 0.0625) * (1 + 2.0 ** -22) + 2.0 ** -20
        if h < 16:
            assert h == math.ceil((R * 1.0625 + 0.0625) * 2 ** 20) / 2 ** 20


@pytest.mark.gpu
@pytest.mark.parametrize("precision,area,slope", [("mixed", 1e-4, 1e-3), ("fp64", 1e-9, 1e-9)])
@pytest.mark.parametrize("big,shell", [(15.0, 20), (17.3, 50), (33.1, 90), (71.9, 60), (40.7, 57)])
def test_large_balls(orc, big, shell, precision, area, slope):
    """A large ball with small ones around it, whose half-spaces leave corners of the cube in place; more
    than 58 neighbours, or 64 vertices, take the large pass, and a cell of more than 128 vertices (90
    small balls: 2 * 96 - 4) is refused.  Areas relative to the atom's sphere, gradients to 2 pi times
    the large radius: the mixed form's bounds, and for FP64 rounding (1.1e-16) times 5 operations in
    each of 180 terms, with triple points whose height is 1e-4 of the radius."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import api
    rng = np.random.default_rng(shell)
    u = rng.normal(size=(shell, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    x = np.concatenate([[[0.01, -0.02, 0.03]], u * (big + rng.uniform(-1.0, 1.5, (shell, 1)))])
    r = np.concatenate([[big - P], rng.uniform(1.2, 2.0, shell)])
    xs, rs = torch.as_tensor(x, device="cuda"), torch.as_tensor(r, device="cuda")
    a, g = torch.empty_like(rs), torch.empty_like(xs)
    ctx = api.Context(precision=precision)
    ctx.compute(xs, rs, a, g)
    if 2 * (shell + 6) - 4 > 128:
        assert ctx.status_code() == 3 and torch.isnan(a[0])
        ctx.close()
        return
    ctx.status_sync()
    rec = ctx.export_complex(xs, rs).cpu().numpy()
    ctx.close()
    ra, _, rg = orc.sasa(x, r)
    R = r + P
    assert np.all(np.abs(a.cpu().numpy() - ra) <= area * 4 * np.pi * R * R)
    assert np.all(np.abs(g.cpu().numpy() - rg) <= slope * 2 * np.pi * R.max())
    o = orc.Oracle(x, r)
    for d in range(4):
        got = {tuple(int(v) for v in row[1:] if v >= 0) for row in rec if (row[1:] >= 0).sum() == d + 1}
        assert got == {tuple(int(v) for v in np.atleast_1d(s)) for s in o.simplices(d)}
