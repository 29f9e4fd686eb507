"""The work that users of this library have it do, as measurable cases.

Every case calls a public entry point on molecule-shaped inputs: the globules, RNA mimics and
capsid shells of ``paper_2401_10462_gb300.inputs``, at sizes between a small peptide and the
1,000,000-atom capsid.  ``exact`` gives the same quantities in float64 from the definition
alone: the exposed area of every ball by the boundary arcs of its covering circles, the
gradients by the motion of those arcs, the volumes by the faces of the power cells.
"""
import math

import numpy as np
import torch

from paper_2401_10462_gb300 import api, autograd, inputs

PROBE = 1.4
DEV = "cuda:0"


def listed():
    return [
        # one energy-and-force evaluation of a mini-protein, the smallest molecule in use: a
        # simulation or a minimiser makes thousands of them one after another
        {"name": "peptide_304", "op": "sasa", "kind": "globule", "n": 304, "precision": "mixed"},
        # the common case: one protein of a few hundred residues, areas and gradient
        {"name": "protein_5000", "op": "sasa", "kind": "globule", "n": 5000, "precision": "mixed"},
        # the same protein where every term is wanted in double precision (reference energies)
        {"name": "protein_5000_fp64", "op": "sasa", "kind": "globule", "n": 5000, "precision": "fp64"},
        # an RNA fragment in double precision, odd size, more than one wave of atoms
        {"name": "rna_13007_fp64", "op": "sasa", "kind": "rna", "n": 13007, "precision": "fp64"},
        # the nonpolar energy of a large protein and its forces through autograd
        {"name": "energy_backward_20003", "op": "energy", "kind": "globule", "n": 20003, "precision": "mixed"},
        # analysis of a long nucleic acid: areas only, no gradient
        {"name": "areas_rna_49999", "op": "areas", "kind": "rna", "n": 49999, "precision": "mixed"},
        # a whole virus capsid in one solve, the largest input in use
        {"name": "capsid_1000000", "op": "sasa", "kind": "shell", "n": 1000000, "precision": "mixed"},
        # consecutive simulation steps with neighbour lists kept between them
        {"name": "md_steps_20000", "op": "md", "kind": "globule", "n": 20000, "frames": 4, "precision": "mixed"},
        # a serving batch: molecules of mixed sizes and kinds with resident neighbour lists
        {"name": "serving_batch_20", "op": "batch", "kind": "mix", "n": 50000, "molecules": 20, "precision": "mixed"},
        # molecular volumes of a protein and the gradient of a weighted sum of them
        {"name": "volume_5000", "op": "volume", "kind": "globule", "n": 5000, "precision": "mixed"},
        # the numerical cross-check of the areas: 960 points per atom
        {"name": "shrake_rupley_5000", "op": "sr", "kind": "globule", "n": 5000, "points": 960, "precision": "mixed"},
        # a host program (an MD engine on the CPU) calling with its own pinned buffers
        {"name": "host_2003", "op": "host", "kind": "globule", "n": 2003, "precision": "mixed"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sasa", "sasa", "sasa", "energy", "areas", "md", "batch", "volume", "sr", "host"])
    kind = rng.choice(["globule", "rna"])
    precision = "mixed"
    if op == "sasa":
        kind = rng.choice(["globule", "rna", "shell"])
        if kind != "shell" and rng.random() < 0.4:
            precision = "fp64"
    n = {"sasa": lambda: _logint(rng, 10000, 400000) if kind == "shell" else _logint(rng, 200, 20000),
         "energy": lambda: _logint(rng, 300, 25000),
         "areas": lambda: _logint(rng, 1000, 50000 if kind == "rna" else 25000),
         "md": lambda: _logint(rng, 1000, 25000),
         "batch": lambda: 50000,
         "volume": lambda: _logint(rng, 300, 10000),
         "sr": lambda: _logint(rng, 300, 10000),
         "host": lambda: _logint(rng, 200, 20000)}[op]()
    case = {"op": op, "kind": "mix" if op == "batch" else kind, "n": n, "precision": precision}
    if op == "md":
        case["frames"] = rng.randint(2, 6)
    if op == "batch":
        case["molecules"] = _logint(rng, 4, 32)
    if op == "sr":
        case["points"] = _logint(rng, 92, 1500)
    return case


# ------------------------------------------------------------------ inputs
_bases = {}


def _base(kind, n):
    """One generated molecule of this kind and size (placing the atoms of a large one takes
    seconds, so that it is done once per process)."""
    if (kind, n) not in _bases:
        _bases[kind, n] = inputs.make(kind, n, 0)
    return _bases[kind, n]


def _molecule(kind, n, seed):
    """coords (n, 3), radii (n) float64 on the device: a newly generated molecule, or, above
    6,000 atoms, one of that size turned at random with every atom displaced by N(0, 0.03 A)."""
    if n <= 6000 or kind == "rna":
        m = {"globule": inputs.globule, "rna": inputs.rna, "shell": inputs.shell}[kind](n, seed)
        return torch.as_tensor(m.coords, device=DEV), torch.as_tensor(m.radii, device=DEV)
    m = _base(kind, n)
    rng = np.random.default_rng(seed)
    q, r = np.linalg.qr(rng.normal(size=(3, 3)))
    q = torch.as_tensor(q * np.sign(np.diag(r)), device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.as_tensor(m.coords, device=DEV) @ q
    x = x + 0.03 * torch.randn(x.shape, generator=gen, device=DEV, dtype=torch.float64)
    return x.contiguous(), torch.as_tensor(m.radii, device=DEV)


def _frames(case, seed):
    """`frames` consecutive positions of one molecule (0.01 A per coordinate and step)."""
    x, r = _molecule(case["kind"], case["n"], seed)
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    xs = [x]
    for _ in range(case["frames"] - 1):
        xs.append(xs[-1] + 0.01 * torch.randn(x.shape, generator=gen, device=DEV, dtype=torch.float64))
    return xs, r


def _mixture(case, seed):
    """offsets, coords, radii of a batch: sizes log-uniform in [300, n], 70 % globules (the
    atoms of a 50,000-atom globule nearest to a random centre), 30 % RNA mimics.  The sizes
    are those of the case, whatever the seed."""
    sizes_rng = np.random.default_rng(977 + case["molecules"])
    rng = np.random.default_rng(seed)
    xs, rs = [], []
    for _ in range(case["molecules"]):
        n = int(round(math.exp(sizes_rng.uniform(math.log(300), math.log(case["n"])))))
        if sizes_rng.random() < 0.3:
            x, r = _molecule("rna", n, int(rng.integers(1 << 30)))
        else:
            big = _base("globule", 50000)
            c = big.coords[int(rng.integers(big.n))]
            near = np.argsort(((big.coords - c) ** 2).sum(1), kind="stable")[:n]
            near.sort()
            x = torch.as_tensor(big.coords[near], device=DEV)
            r = torch.as_tensor(big.radii[near], device=DEV)
            gen = torch.Generator(device=DEV).manual_seed(int(rng.integers(1 << 30)))
            x = x + 0.03 * torch.randn(x.shape, generator=gen, device=DEV, dtype=torch.float64)
        xs.append(x)
        rs.append(r)
    off = np.concatenate([[0], np.cumsum([len(r) for r in rs])]).astype(np.int64)
    return off, torch.cat(xs).contiguous(), torch.cat(rs).contiguous()


def _weights(n, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed + 2)
    return 0.5 + torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)


# ------------------------------------------------------------------ what a program keeps
_contexts = {}


def _context(precision):
    """The library context that a program keeps for its calls in this precision."""
    if precision not in _contexts:
        _contexts[precision] = api.Context(precision=precision)
    return _contexts[precision]


def prepare(case, seed):
    op, n = case["op"], case["n"]
    f64 = dict(dtype=torch.float64, device=DEV)
    s = {"case": case, "op": op}
    if op == "batch":
        s["off"], s["x"], s["r"] = _mixture(case, seed)
        n = int(s["off"][-1])
        s["ctx"] = api.Context(precision=case["precision"], skin=1.0)
        s["arena"] = api.Arena(n)
        s["areas"], s["grad"] = torch.empty(n, **f64), torch.empty((n, 3), **f64)
        return s
    if op == "md":
        s["xs"], s["r"] = _frames(case, seed)
        s["ctx"] = api.Context(precision=case["precision"], skin=1.0)
        s["areas"] = [torch.empty(n, **f64) for _ in s["xs"]]
        s["grad"] = [torch.empty((n, 3), **f64) for _ in s["xs"]]
        return s
    s["x"], s["r"] = _molecule(case["kind"], n, seed)
    s["ctx"] = _context(case["precision"])
    if op == "host":
        for k, shape in (("x", (n, 3)), ("r", (n,)), ("areas", (n,)), ("grad", (n, 3))):
            t = torch.empty(shape, dtype=torch.float64, pin_memory=True)
            if k in ("x", "r"):
                t.copy_(s[k])
            s["pinned_" + k], s[k] = t, t.numpy()
        return s
    s["areas"], s["grad"] = torch.empty(n, **f64), torch.empty((n, 3), **f64)
    if op == "energy":
        s["x"].requires_grad_(True)
    if op == "volume":
        s["w"], s["vol"] = _weights(n, seed), torch.empty(n, **f64)
    if op == "sr":
        s["pts"] = torch.as_tensor(inputs.sphere_points(case["points"]), device=DEV)
        s["exposed"] = torch.empty(n, dtype=torch.int32, device=DEV)
    return s


def run(s):
    op, ctx = s["op"], s["ctx"]
    if op == "sasa":
        ctx.compute(s["x"], s["r"], s["areas"], s["grad"])
        return {"areas": s["areas"], "grad": s["grad"]}
    if op == "energy":
        e, areas = autograd.nonpolar_energy(s["x"], s["r"], precision=s["case"]["precision"])
        (g,) = torch.autograd.grad(e, s["x"])
        return {"energy": e.detach(), "areas": areas.detach(), "grad": g}
    if op == "areas":
        return {"areas": autograd.sasa_areas(s["x"], s["r"], precision=s["case"]["precision"])}
    if op == "md":
        for x, a, g in zip(s["xs"], s["areas"], s["grad"]):
            ctx.compute(x, s["r"], a, g)
        return {"areas": s["areas"], "grad": s["grad"]}
    if op == "batch":
        ctx.compute_batch_resident(s["off"], s["x"], s["r"], s["areas"], s["grad"], arena=s["arena"],
                                   arena_base=s["off"][:-1])
        return {"areas": s["areas"], "grad": s["grad"]}
    if op == "volume":
        ctx.compute_volume_vjp(s["x"], s["r"], s["w"], s["areas"], s["vol"], s["grad"])
        return {"areas": s["areas"], "volumes": s["vol"], "grad": s["grad"]}
    if op == "sr":
        ctx.compute_sr(s["x"], s["r"], s["pts"], s["areas"], s["exposed"])
        return {"areas": s["areas"], "exposed": s["exposed"]}
    if op == "host":
        ctx.compute_host(s["x"], s["r"], out=(s["areas"], s["grad"]))
        return {"areas": s["areas"], "grad": s["grad"]}
    raise ValueError(op)


def work(case):
    """Inputs read once, outputs written once; operations of the certified cell vertices (520
    for each of 26.5 star tetrahedra per atom) and of the area terms (3,750 per atom, three
    times that with the gradient); 9 for each test of a point against a neighbour (45)."""
    op, n, calls = case["op"], case["n"], case.get("frames", 1)
    if op == "batch":
        rng = np.random.default_rng(977 + case["molecules"])
        n = 0
        for _ in range(case["molecules"]):
            n += int(round(math.exp(rng.uniform(math.log(300), math.log(case["n"])))))
            rng.random()
    if op == "sr":
        return {"bytes": n * (32 + 8 + 4) + 12 * case["points"], "flops": 9.0 * 45 * case["points"] * n}
    if op == "areas":
        return {"bytes": 40.0 * n, "flops": (13800.0 + 3750) * n}
    if op == "volume":
        return {"bytes": (32.0 + 8 + 8 + 8 + 24) * n, "flops": (13800.0 + 3750 + 5000) * n}
    return {"bytes": 64.0 * n * calls, "flops": (13800.0 + 11250) * n * calls}


# ------------------------------------------------------------------ float64 from the definition
def _neighbours(x, R, mol=None):
    """(n, K) indices of the atoms whose balls overlap each ball, -1 where there are fewer."""
    n = len(x)
    cell = 2 * float(R.max()) + 1e-6
    lo = x.min(0).values
    c = ((x - lo) / cell).long()
    dims = c.max(0).values + 3
    m = mol if mol is not None else torch.zeros(n, dtype=torch.long, device=x.device)
    cid = (((m * dims[0] + c[:, 0] + 1) * dims[1] + c[:, 1] + 1) * dims[2]) + c[:, 2] + 1
    key, order = torch.sort(cid)
    best = []
    for i0 in range(0, n, 50000):
        i = torch.arange(i0, min(n, i0 + 50000), device=x.device)
        cand, good = [], []
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                first = cid[i] + (dx * dims[1] + dy) * dims[2]
                a, b = torch.searchsorted(key, first - 1), torch.searchsorted(key, first + 1, right=True)
                k = a[:, None] + torch.arange(int((b - a).max()), device=x.device)
                ok = k < b[:, None]
                j = order[k.clamp(max=n - 1)]
                d2 = ((x[j] - x[i][:, None]) ** 2).sum(-1)
                cand.append(j)
                good.append(ok & (j != i[:, None]) & (d2 < (R[j] + R[i][:, None]) ** 2))
        cand, good = torch.cat(cand, 1), torch.cat(good, 1)
        k = int(good.sum(1).max())
        where = torch.argsort(~good, dim=1, stable=True)[:, :k]
        best.append(torch.where(good.gather(1, where), cand.gather(1, where), torch.full_like(where, -1)))
    k = max(1, max(b.shape[1] for b in best))
    return torch.cat([torch.nn.functional.pad(b, (0, k - b.shape[1]), value=-1) for b in best])


def _solid(a, b, c):
    """Signed solid angle of the triangle of unit vectors a, b, c."""
    num = (a * torch.linalg.cross(b, c)).sum(-1)
    return 2 * torch.atan2(num, 1 + (a * b).sum(-1) + (b * c).sum(-1) + (c * a).sum(-1))


def _surface(x, R, w, mol=None, volume=False):
    """Exposed areas A_i and d(sum_i w_i A_i)/dx; with `volume`: A_i, the volumes V_i of the
    balls cut by their power bisectors, and d(sum_i w_i V_i)/dx."""
    n = len(x)
    nb = _neighbours(x, R, mol)
    A = torch.zeros_like(R)
    V = torch.zeros_like(R)
    g = torch.zeros_like(x)
    step = max(1, int((2e6 if volume else 4e7) / nb.shape[1] ** (3 if volume else 2)))
    for i0 in range(0, n, step):
        i = torch.arange(i0, min(n, i0 + step), device=x.device)
        J = nb[i]
        Ri, Rj = R[i][:, None], R[J.clamp(min=0)]
        q = x[J.clamp(min=0)] - x[i][:, None]
        d = q.norm(dim=-1)
        have = J >= 0
        d = torch.where(have, d, torch.ones_like(d))
        t = (d * d + (Ri - Rj) * (Ri + Rj)) / (2 * d)
        inside = (have & (t <= -Ri)).any(1)          # the whole ball lies in another one
        cut = have & (t.abs() < Ri)                  # the circle of ball j on sphere i
        nrm = q / d[..., None]
        r = torch.where(cut, (Ri * Ri - t * t).clamp(min=1e-300).sqrt(), torch.ones_like(t))
        axis = torch.nn.functional.one_hot(nrm.abs().argmin(-1), 3).to(x.dtype)
        e1 = torch.linalg.cross(nrm, axis)
        e1 = e1 / e1.norm(dim=-1, keepdim=True)
        e2 = torch.linalg.cross(nrm, e1)
        # circle j (rows) against ball k (columns): the covered arc [phi - al, phi + al]
        gjk = torch.einsum("aji,aki->ajk", nrm, nrm)
        u1 = torch.einsum("aji,aki->ajk", e1, nrm)
        u2 = torch.einsum("aji,aki->ajk", e2, nrm)
        s = (u1 * u1 + u2 * u2).sqrt()
        c = (t[:, None, :] - t[:, :, None] * gjk) / (r[..., None] * s).clamp(min=1e-300)
        k = J.shape[1]
        other = cut[:, :, None] & cut[:, None, :] & ~torch.eye(k, dtype=torch.bool, device=x.device)
        full = (other & (c <= -1)).any(2)
        al = torch.acos(c.clamp(-1, 1))
        part = other & (c.abs() < 1)
        b0 = torch.remainder(torch.atan2(u2, u1) - al, 2 * math.pi)
        b0 = torch.where(part, b0, torch.full_like(b0, math.inf))
        b0, o = torch.sort(b0, dim=2)
        b1 = b0 + 2 * al.gather(2, o)
        any_part = part.any(2)
        # the exposed arcs: from the largest end so far to the next start
        end = torch.cummax(torch.where(b0.isfinite(), b1, torch.full_like(b1, -math.inf)), dim=2).values
        end = torch.maximum(end, end[:, :, -1:] - 2 * math.pi)      # an arc that runs past the turn
        first = torch.where(any_part, b0[:, :, 0], torch.zeros_like(b0[:, :, 0]))
        nxt = torch.cat([b0[:, :, 1:], torch.full_like(b0[:, :, :1], math.inf)], 2)
        nxt = torch.where(nxt.isfinite(), nxt, (first + 2 * math.pi)[..., None].expand_as(nxt))
        nxt = torch.minimum(nxt, (first + 2 * math.pi)[..., None])
        gap = b0.isfinite() & (nxt > end)
        a0 = torch.where(gap, end, torch.zeros_like(end))
        a1 = torch.where(gap, nxt, torch.zeros_like(end))
        whole = cut & ~any_part & ~full
        a1[:, :, 0] = torch.where(whole, torch.full_like(a1[:, :, 0], 2 * math.pi), a1[:, :, 0])
        arc = (gap | (whole[..., None] & (torch.arange(k, device=x.device) == 0))) & (cut & ~full)[..., None]
        a0, a1 = torch.where(arc, a0, torch.zeros_like(a0)), torch.where(arc, a1, torch.zeros_like(a1))
        dphi = (a1 - a0).sum(2)
        ic = (torch.sin(a1) - torch.sin(a0)).sum(2)      # integrals of cos and sin over the arcs
        is_ = (torch.cos(a0) - torch.cos(a1)).sum(2)
        # area, modulo the sphere: minus what the arcs (counter-clockwise about n_j) enclose
        ai, aj, ak = torch.nonzero(arc & ~(whole[..., None]), as_tuple=True)
        tj, rj, Rs = t[ai, aj][:, None], r[ai, aj][:, None], R[i][ai][:, None]
        def at(phi):
            p = torch.cos(phi)[:, None] * e1[ai, aj] + torch.sin(phi)[:, None] * e2[ai, aj]
            return (tj * nrm[ai, aj] + rj * p) / Rs
        # each arc in three pieces, so that the triangles stay well away from a half turn
        p0, p1 = a0[ai, aj, ak], a1[ai, aj, ak]
        pole = torch.tensor([0.36, -0.48, 0.8], dtype=x.dtype, device=x.device).expand(len(ai), 3)
        enclosed = torch.zeros_like(R[i])
        for h in range(3):
            f0, f1 = p0 + (p1 - p0) * (h / 3), p0 + (p1 - p0) * ((h + 1) / 3)
            v0, v1, m = at(f0), at(f1), nrm[ai, aj]
            sector = (f1 - f0) * (1 - tj[:, 0] / Rs[:, 0])
            enclosed.index_add_(0, ai, _solid(pole, v0, v1) + sector - _solid(m, v0, v1))
        enclosed += torch.where(whole, 2 * math.pi * (1 - t / Ri), torch.zeros_like(t)).sum(1)
        om = torch.remainder(-enclosed, 4 * math.pi)
        om = torch.where(om > 4 * math.pi - 1e-6, om - 4 * math.pi, om)
        om = torch.where(arc.flatten(1).any(1), om, torch.where(cut.any(1), torch.zeros_like(om), torch.full_like(om, 4 * math.pi)))
        om = torch.where(inside, torch.zeros_like(om), om)
        A[i] = R[i] ** 2 * om
        live = (cut & ~inside[:, None])[..., None]
        ring = ic[..., None] * e1 + is_[..., None] * e2
        if not volume:
            f = -(Ri / d)[..., None] * ((t - d)[..., None] * dphi[..., None] * nrm + r[..., None] * ring)
            f = torch.where(live, f, torch.zeros_like(f)) * w[i][:, None, None]
            g.index_add_(0, J.clamp(min=0).reshape(-1), f.reshape(-1, 3))
            g[i] -= f.sum(1)
            continue
        # the face of bisector j inside the ball: its disk cut by the other bisectors' lines
        cl = torch.where(other, (t[:, None, :] - t[:, :, None] * gjk) / s.clamp(min=1e-300), torch.full_like(s, math.inf))
        ux, uy = u1 / s.clamp(min=1e-300), u2 / s.clamp(min=1e-300)
        half = (r[..., None] ** 2 - cl * cl)
        on = other & (half > 0)
        half = half.clamp(min=0).sqrt()
        # the point of line k at parameter p: cl u + p v, v = (-uy, ux); bisector l keeps u_l . y <= cl_l
        dot = torch.einsum("ajk,ajl->ajkl", ux, ux) + torch.einsum("ajk,ajl->ajkl", uy, uy)
        crs = torch.einsum("ajk,ajl->ajkl", ux, uy) - torch.einsum("ajk,ajl->ajkl", uy, ux)
        use = other[:, :, None, :] & ~torch.eye(k, dtype=torch.bool, device=x.device)
        lim = (cl[:, :, None, :] - torch.where(other, cl, torch.zeros_like(cl))[..., None] * dot) / crs
        inf = torch.full_like(lim, math.inf)
        hi = torch.where(use & (crs > 0), lim, inf).amin(-1)
        lw = torch.where(use & (crs < 0), lim, -inf).amax(-1)
        hi, lw = torch.minimum(hi, half), torch.maximum(lw, -half)
        on &= (hi > lw) & (cut & ~inside[:, None])[..., None]
        clz = torch.where(on, cl, torch.zeros_like(cl))
        hi, lw = torch.where(on, hi, torch.zeros_like(hi)), torch.where(on, lw, torch.zeros_like(lw))
        tri = 0.5 * clz * (hi - lw)
        sec = 0.5 * r * r * dphi
        sf = torch.where(live[..., 0], tri.sum(2) + sec, torch.zeros_like(sec))
        mid = 0.5 * (hi + lw)
        m1 = (tri * (2.0 / 3) * (clz * ux - mid * uy)).sum(2) + r ** 3 / 3 * ic
        m2 = (tri * (2.0 / 3) * (clz * uy + mid * ux)).sum(2) + r ** 3 / 3 * is_
        mf = (sf * t)[..., None] * nrm + m1[..., None] * e1 + m2[..., None] * e2
        mf = torch.where(live, mf, torch.zeros_like(mf))
        # a ball wholly beyond a bisector, or one with no circle at all, keeps what its area says
        V[i] = torch.where(inside, torch.zeros_like(A[i]), (R[i] * A[i] + (t * sf).sum(1)) / 3)
        wk = torch.where(J >= 0, w[J.clamp(min=0)], torch.zeros_like(t))
        g[i] = -w[i][:, None] * (sf[..., None] * nrm).sum(1) + (((w[i][:, None] - wk) / d)[..., None] * mf).sum(1)
    return (A, V, g) if volume else (A, g)


def exact(case, seed):
    op, n = case["op"], case["n"]
    if op == "md":
        xs, r = _frames(case, seed)
        got = [_surface(x, r + PROBE, torch.ones_like(r)) for x in xs]
        return {"areas": [a for a, _ in got], "grad": [g for _, g in got]}
    if op == "batch":
        off, x, r = _mixture(case, seed)
        mol = torch.repeat_interleave(torch.arange(len(off) - 1, device=DEV), torch.as_tensor(np.diff(off), device=DEV))
        a, g = _surface(x, r + PROBE, torch.ones_like(r), mol)
        return {"areas": a, "grad": g}
    x, r = _molecule(case["kind"], n, seed)
    if op == "sr":
        return None          # counts of points (whole numbers) and fixed multiples of them
    R = r + PROBE
    if op == "volume":
        a, v, g = _surface(x, R, _weights(n, seed), volume=True)
        return {"areas": a, "volumes": v, "grad": g}
    a, g = _surface(x, R, torch.full_like(R, autograd.GAMMA) if op == "energy" else torch.ones_like(R))
    if op == "energy":
        return {"energy": autograd.GAMMA * a.sum(), "areas": a, "grad": g}
    if op == "areas":
        return {"areas": a}
    return {"areas": a, "grad": g}
