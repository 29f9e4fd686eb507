"""The check of a cell's structure (csrc/dsasa_cell.cuh, compiled for the host by g++), as the clipping
makes it of every cell whose signs were resolved exactly: a consistent cell passes, a cell with any byte changed does
not, and no cell that passes has a face whose walk fails to close."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2401_10462_gb300", "csrc")
SRC = os.path.join(HERE, "cellcheck.cpp")
SO = os.path.join(ROOT, "paper_2401_10462_gb300", "_build", "libcellcheck.so")


@pytest.fixture(scope="module")
def lib():
    os.makedirs(os.path.dirname(SO), exist_ok=True)
    deps = [SRC, os.path.join(CSRC, "dsasa_cell.cuh"), os.path.join(CSRC, "dsasa_math.cuh")]
    if not os.path.exists(SO) or os.path.getmtime(SO) < max(os.path.getmtime(d) for d in deps):
        tmp = SO + f".tmp{os.getpid()}"
        subprocess.check_call(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-o", tmp, SRC])
        os.replace(tmp, SO)
    return ctypes.CDLL(SO)


def _cell(planes, seed):
    """A simple polytope with `planes` faces, as its dual triangulation of a sphere: each new point is
    put into a triangle (4 planes: a tetrahedron), then random edges are flipped."""
    rng = np.random.default_rng(seed)
    tri = [(0, 1, 2), (0, 3, 1), (1, 3, 2), (2, 3, 0)]
    for m in range(4, planes):
        a, b, c = tri.pop(rng.integers(len(tri)))
        tri += [(a, b, m), (b, c, m), (c, a, m)]
    for _ in range(4 * planes):
        edge = {(t[k], t[(k + 1) % 3]): (i, t[(k + 2) % 3]) for i, t in enumerate(tri) for k in range(3)}
        (a, b) = list(edge)[rng.integers(len(edge))]
        (i, c), (j, d) = edge[a, b], edge[b, a]
        if (c, d) not in edge and (d, c) not in edge and c != d:
            tri[i], tri[j] = (a, d, c), (d, b, c)
    edge = {(t[k], t[(k + 1) % 3]): i for i, t in enumerate(tri) for k in range(3)}
    assert len(edge) == 3 * len(tri)
    adj = [tuple(edge[t[(k + 1) % 3], t[k]] for k in range(3)) for t in tri]
    return np.array(tri), np.array(adj)


def _disagreeing(lib, v, adj):
    w = [np.ascontiguousarray(x[:, 0] | x[:, 1] << 8 | x[:, 2] << 16, dtype=np.uint32) for x in (v, adj)]
    return lib.cc_disagreeing(*(x.ctypes.data_as(ctypes.POINTER(ctypes.c_uint)) for x in w), len(v))


def _walks_close(v, adj):
    for t0 in range(len(v)):
        for a in v[t0]:
            t = t0
            for _ in range(len(v) + 1):
                k = list(v[t]).index(a) if a in v[t] else 2
                t = adj[t][k]
                if t == t0:
                    break
            else:
                return False
    return True


@pytest.mark.parametrize("planes", [4, 6, 12, 19, 34])
def test_consistent_cells_pass_and_changed_ones_do_not(lib, planes):
    v, adj = _cell(planes, planes)
    n = len(v)
    assert n == 2 * planes - 4 and _disagreeing(lib, v, adj) == 0 and _walks_close(v, adj)
    rng = np.random.default_rng(1)
    for _ in range(300):
        w, b = v.copy(), adj.copy()
        t, k = rng.integers(n), rng.integers(3)
        kind = rng.integers(4)
        if kind == 0:
            b[t, k] = rng.choice([x for x in range(n + 2) if x != adj[t, k]])
        elif kind == 1:
            w[t, k] = rng.choice([x for x in range(planes + 1) if x != v[t, k]])
        elif kind == 2:
            w[t] = w[t][[1, 0, 2]]
        else:
            w[t] = 255     # a dead slot that its neighbours still name
        assert _disagreeing(lib, w, b) > 0, (kind, t, k)


@pytest.mark.parametrize("planes", [5, 8, 14])
def test_no_passing_cell_has_an_open_face(lib, planes):
    """Two neighbours exchanged anywhere: the cell is refused, or every walk closes all the same."""
    v, adj = _cell(planes, planes)
    n = len(v)
    rng = np.random.default_rng(2)
    for _ in range(400):
        b = adj.copy()
        for _ in range(rng.integers(1, 4)):
            (s, j), (t, k) = rng.integers(n, size=2), rng.integers(3, size=2)
            (s, t), (j, k) = (s, j), (t, k)
            b[s, j], b[t, k] = b[t, k], b[s, j]
        assert _disagreeing(lib, v, b) > 0 or _walks_close(v, b)
