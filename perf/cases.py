"""What the library is timed on: its public entry points over the range of sizes and options that programs use.

Every case is one call sequence of a program that uses paper_0903_1949_gb300 (rt.Grid, rt.Batch, rt.Line,
rt.rt_fs_sweep or autograd.solve) on the synthetic atmospheres of inputs.py: the spherical grids with
chi ~ r^-2 and 20 % lognormal noise, and the cylindrical disc.  A grid (the crossing lists of its
characteristics) is what such a program creates once and keeps; opacities, source functions and results
are FP64 arrays on the GPU, as the library takes and gives them.  Results of mixed-precision passes carry
the FP32 rounding of the ray march, and the program here keeps them as FP32.

exact() evaluates the same problem in plain torch FP64: the launch set and the crossings of every line,
the recurrence along each characteristic, the averages, the ALI and Ng updates, the fixed point and its
adjoint, each written out here from their definitions.
"""
import math
import time

import numpy as np
import torch

from paper_0903_1949_gb300 import autograd, rt
from paper_0903_1949_gb300 import inputs as I

# crossing segments per voxel and solid angle, for work() (spherical, cylindrical)
SEGS = (5.9, 2.8)


def _case(name, kind, n, ang, tau, eps, **kw):
    c = dict(kind=kind, coord=I.SPHERICAL, n1=n[0], n2=n[1], n3=n[2], mu=ang[0], phi=ang[1], tau=float(tau),
             eps=float(eps), precision=rt.RT_FP64, lstar=rt.RT_LSTAR_DIAG, steps=4, members=1, tol=1e-8)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    mixed = dict(precision=rt.RT_MIXED)
    disc = dict(coord=I.CYLINDRICAL)
    nn = dict(lstar=rt.RT_LSTAR_NN)
    return [
        # a toy grid of the tests: a handful of ALI iterations, where launches and waits count
        _case("ali_tiny_mixed", "ali", (7, 5, 9), (4, 4), 4.0, 1e-1, **mixed),
        # the small spherical model solved to convergence for a new opacity, all FP64
        _case("solve_sph17_f64", "solve", (17, 9, 17), (8, 8), 4.0, 1e-2),
        # the paper's spherical grid at the benchmark's 32 x 32 solid angles: four mixed ALI iterations and Ng
        _case("ali_sph65_mixed", "ali", (65, 33, 65), (32, 32), 1e2, 1e-4, **mixed),
        # the same iterations all in FP64, with fewer solid angles
        _case("ali_sph65_f64", "ali", (65, 33, 65), (16, 16), 1e2, 1e-4),
        # the cylindrical disc: four mixed ALI iterations and Ng
        _case("ali_cyl65_mixed", "ali", (65, 65, 65), (16, 16), 1e3, 1e-6, **mixed, **disc),
        # one formal solution (J, Lambda*, flux) of a new opacity in mixed precision: a snapshot of a
        # hydrodynamics or post-processing run
        _case("fs_sph65_mixed", "fs", (65, 33, 65), (16, 16), 1e2, 1e-4, **mixed),
        # the same in FP64 on an odd disc grid
        _case("fs_cyl_f64", "fs", (49, 37, 51), (12, 10), 1e2, 1e-4, **disc),
        # angle-resolution study: geometry and formal solution of a solid-angle set, in chunks
        _case("sweep_sph65_mixed", "sweep", (65, 33, 65), (8, 16), 1e1, 1e-4, members=2, **mixed),
        # scattering-dominated model: nearest-neighbour operator of a new opacity and the solve with it
        _case("solve_nn_f64", "solve", (33, 17, 33), (8, 8), 1e2, 1e-4, **nn),
        # gradients of a converged model with respect to chi, eps and B (forward and backward)
        _case("grad_sph33", "grad", (33, 17, 33), (8, 8), 1e1, 1e-1, tol=1e-11),
        # many wavelengths on two grids of uneven size: new opacities, then batched ALI iterations
        _case("batch12_mixed", "batch", (65, 33, 65), (8, 8), 1.0, 1e-3, members=12, **mixed),
        # two-level line, 32 frequencies, nearest-neighbour line operator and Ng
        _case("line32_nn_mixed", "line", (33, 17, 33), (8, 8), 1.0, 1e-4, members=32, **nn, **mixed),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("ali", "ali", "ali", "fs", "solve", "sweep", "grad", "batch", "line"))
    coord = I.CYLINDRICAL if kind in ("ali", "fs", "solve", "sweep") and rng.random() < 0.35 else I.SPHERICAL
    small = kind in ("grad", "line", "solve")  # hundreds of formal solutions a pass, or dozens of operators
    top = 33 if small else 65
    while True:
        n = [_logint(rng, 5, top), _logint(rng, 4, top // 2 + 1), _logint(rng, 5, top)]
        if coord == I.CYLINDRICAL:
            n[1] = _logint(rng, 4, top)
        ang = (2 * _logint(rng, 1, 8), _logint(rng, 3, 16))
        members = {"batch": rng.randint(2, 12), "line": rng.randint(4, 32), "sweep": rng.randint(1, 3)}.get(kind, 1)
        lines = n[0] * n[1] * n[2] * ang[0] * ang[1]
        most = {"sweep": 1.5e7, "batch": 1e8 / members, "line": 3e7 / members}.get(kind, 1.5e6 if small else 4e7)
        if lines <= most:
            break
    prec = rt.RT_MIXED if kind in ("batch", "line") or (kind in ("ali", "fs", "sweep") and rng.random() < 0.5) else rt.RT_FP64
    nn = kind in ("line", "solve") and rng.random() < 0.5
    tau = 1.0 if kind == "batch" else 10.0 ** rng.uniform(-1.0, 1.0 if small else 3.0)
    eps = 10.0 ** rng.uniform(-2.0, -0.5) if small else 10.0 ** rng.uniform(-4.0, -0.5)
    return _case(None, kind, n, ang, tau, eps, coord=coord, precision=prec, members=members,
                 lstar=rt.RT_LSTAR_NN if nn else rt.RT_LSTAR_DIAG, steps=rng.randint(1, 6),
                 tol=1e-11 if kind == "grad" else 1e-8)


# ---- what a program has in hand -------------------------------------------------------------------


def _shapes(case):
    """Grid sizes of a case: a batch has a second, smaller grid."""
    n = (case["n1"], case["n2"], case["n3"])
    return [n, tuple(max(4, q // 2 + 1) for q in n)] if case["kind"] == "batch" else [n]


def _edges(coord, n):
    return I.sph_edges(*n) if coord == I.SPHERICAL else I.cyl_edges(*n)


def _fields(case, n, seed, tau):
    """chi, B of the named laws of inputs.py with 20 % lognormal noise, flat float64 arrays."""
    name = "sph65" if case["coord"] == I.SPHERICAL else "cyl65"
    p = I.make_problem(name, n=n, n_mu=case["mu"], n_phi=case["phi"], tau=tau, eps=case["eps"], noise=0.0)
    chi = p["chi"] * I.lognormal(p["chi"].size, 0.2, seed)
    B = p["B"] * I.lognormal(p["B"].size, 0.2, seed + 1)
    return chi, B


def _inputs(case, seed):
    """Host arrays of a case, the same for the library and for exact()."""
    rng = np.random.default_rng(seed)
    out = dict(members=[], seed=seed)
    shapes = _shapes(case)
    for m in range(case["members"] if case["kind"] == "batch" else 1):
        n = shapes[m % len(shapes)]
        tau = case["tau"] * (10.0 ** rng.uniform(-2.0, 2.0) if case["kind"] == "batch" else 1.0)
        chi, B = _fields(case, n, int(rng.integers(1 << 30)), tau)
        out["members"].append((chi, np.full(chi.size, case["eps"]), B))
    nv = out["members"][0][0].size
    if case["kind"] == "line":  # grey continuum of radial depth 1e-2, the line 1e6 times stronger
        chi = out["members"][0][0]
        out["chi_c"], out["chi_l"] = chi * (1e-2 / case["tau"]), chi * (1e4 / case["tau"])
    if case["kind"] == "grad":
        out["g"] = [rng.standard_normal(nv), rng.standard_normal(nv), rng.standard_normal((nv, 3))]
    return out


def _cuda(a):
    return torch.as_tensor(a, dtype=torch.float64).cuda().contiguous()


def prepare(case, seed):
    x = _inputs(case, seed)
    dirs, wts = I.angle_set(case["mu"], case["phi"])
    coord = case["coord"]
    bc = I.CORE_B if coord == I.SPHERICAL else I.TRANSPARENT
    st = dict(case=case, chi=[_cuda(m[0]) for m in x["members"]], eps=[_cuda(m[1]) for m in x["members"]],
              B=[_cuda(m[2]) for m in x["members"]])
    shapes = _shapes(case)
    if case["kind"] == "sweep":
        st.update(edges=_edges(coord, shapes[0]), dirs=dirs, wts=wts, bc=bc, S=st["B"][0].clone())
    else:
        st["grids"] = [rt.Grid(coord, _edges(coord, n), dirs, wts, inner_bc=bc, precision=case["precision"],
                               use_lstar=case["lstar"] if case["kind"] == "solve" else rt.RT_LSTAR_DIAG)
                       for n in shapes]
    if case["kind"] == "ali":
        st["grids"][0].set_opacity(st["chi"][0], st["eps"][0], st["B"][0])
        st["S"] = st["B"][0].clone()
    if case["kind"] == "batch":
        st["batch"] = rt.Batch(st["grids"], [m % 2 for m in range(case["members"])])
    if case["kind"] == "line":
        phi, wq = I.line_profile(case["members"])
        st["line"] = rt.Line(st["grids"][0], phi, wq, use_lstar=case["lstar"], ng=True)
        st["chi_c"], st["chi_l"] = _cuda(x["chi_c"]), _cuda(x["chi_l"])
    if case["kind"] == "grad":
        st["g"] = [_cuda(g) for g in x["g"]]
        for k in ("chi", "eps", "B"):
            st[k][0].requires_grad_(True)
    st["out"] = [torch.empty((6 * c.numel(),), dtype=torch.float64, device="cuda") for c in st["chi"]]
    return st


def _keep(case, v):
    return v.float() if case["precision"] == rt.RT_MIXED else v


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "grad":
        g = st["grids"][0]
        leaf = [st[k][0] for k in ("chi", "eps", "B")]
        S, J, F = autograd.solve(g, *leaf, tol=case["tol"], adj_tol=case["tol"])
        d = torch.autograd.grad((S, J, F), leaf, st["g"])
        return dict(S=S.detach(), J=J.detach(), F=F.detach(), dchi=d[0], deps=d[1], dB=d[2])
    nv = [c.numel() for c in st["chi"]]
    buf = [(o[:n], o[n:2 * n], o[2 * n:3 * n], o[3 * n:]) for o, n in zip(st["out"], nv)]
    if kind == "batch":
        b = st["batch"]
        for m in range(case["members"]):
            b.set_member(m, st["chi"][m], st["eps"][m], st["B"][m])
        for _ in range(case["steps"]):
            b.ali_step()
        res = {}
        for m in range(case["members"]):
            res["S%d" % m] = _keep(case, rt.rt_batch_get(b.h, m, 0, nv[m], buf[m][0]))
            res["J%d" % m] = _keep(case, rt.rt_batch_get(b.h, m, 1, nv[m], buf[m][1]))
        return res
    S, J, L, F = buf[0]
    if kind == "line":
        ln = st["line"]
        ln.set(st["chi_c"], st["chi_l"], st["eps"][0], st["B"][0])
        for _ in range(case["steps"]):
            ln.step()
        rt.rt_line_get(ln.h, 0, nv[0], S)
        rt.rt_line_get(ln.h, 1, nv[0], J)
        return dict(S=_keep(case, S), J=_keep(case, J))
    if kind == "sweep":
        per = -(-len(st["wts"]) // case["members"])
        rt.rt_fs_sweep(case["coord"], st["edges"], st["dirs"], st["wts"], st["chi"][0], st["S"], st["B"][0], per,
                       precision=case["precision"], inner_bc=st["bc"], J=J, F=F)
        return dict(J=_keep(case, J), F=_keep(case, F))
    g = st["grids"][0]
    if kind == "ali":
        g.set_S(st["S"])
        for _ in range(case["steps"]):
            g.ali_step()
        g.S(S)
        g.J(J)
        return dict(S=_keep(case, S), J=_keep(case, J))
    g.set_opacity(st["chi"][0], st["eps"][0], st["B"][0])
    if kind == "fs":
        g.formal_solution()
        g.J(J)
        g.Lstar(L)
        g.flux(F)
        return dict(J=_keep(case, J), L=_keep(case, L), F=_keep(case, F))
    g.solve(case["tol"], 2000)  # kind == "solve"
    g.S(S)
    g.J(J)
    return dict(S=_keep(case, S), J=_keep(case, J))


def work(case):
    """Each crossing read once per formal solution (voxel id and path length: 8 bytes in FP32, 12 in FP64)
    with a voxel's fields read and its results written once; the recurrence of a segment (two products with
    sums of its own, the optical depth, an exponential and its weights) at 20 operations."""
    nv = sum(n[0] * n[1] * n[2] for n in _shapes(case)) / len(_shapes(case))
    seg = nv * case["mu"] * case["phi"] * SEGS[case["coord"]]
    per = 8 if case["precision"] == rt.RT_MIXED else 12
    sols = {"ali": case["steps"], "fs": 1, "sweep": 1, "batch": case["members"] * (case["steps"] + 1),
            "line": case["members"] * (case["steps"] + 1), "solve": 30, "grad": 100}[case["kind"]]
    return {"bytes": sols * (per * seg + 48 * nv), "flops": 20 * sols * seg}


# ---- the same in plain torch FP64 -----------------------------------------------------------------

INF = float("inf")


class _Lines:
    """Straight lines through the centres of voxels (index v) in directions d (N x 3) of a grid."""

    def __init__(self, coord, edges, dev):
        self.coord, self.dev = coord, dev
        self.n = [len(e) - 1 for e in edges]
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.e = [t(np.asarray(e)) for e in edges]
        mid = lambda e: [0.5 * (e[q] + e[q + 1]) for q in range(len(e) - 1)]  # noqa: E731
        ph = edges[2] if coord == I.SPHERICAL else edges[1]
        self.nphi = len(ph) - 1
        self.cp, self.sp = t([math.cos(p) for p in ph[:-1]]), t([math.sin(p) for p in ph[:-1]])
        self.cpm, self.spm = t([math.cos(p) for p in mid(ph)]), t([math.sin(p) for p in mid(ph)])
        if coord == I.SPHERICAL:
            self.ct = t([math.cos(p) for p in edges[1]])
            self.ctm, self.stm = t([math.cos(p) for p in mid(edges[1])]), t([math.sin(p) for p in mid(edges[1])])

    def ijk(self, v):
        n1, n2, n3 = self.n
        return v // (n2 * n3), (v // n3) % n2, v % n3

    def centre(self, v):
        i, j, k = self.ijk(v)
        r = 0.5 * (self.e[0][i] + self.e[0][i + 1])
        if self.coord == I.SPHERICAL:
            w = r * self.stm[j]
            return w * self.cpm[k], w * self.spm[k], r * self.ctm[j]
        return r * self.cpm[j], r * self.spm[j], 0.5 * (self.e[2][k] + self.e[2][k + 1])

    def starts(self, v, d):
        """Masks: the line's direction enters the domain at voxel v, or leaves the core there."""
        i, j, k = self.ijk(v)
        if self.coord == I.SPHERICAL:
            dot = (d[:, 0] * (self.stm[j] * self.cpm[k]) + d[:, 1] * (self.stm[j] * self.spm[k])) + d[:, 2] * self.ctm[j]
            return (i == self.n[0] - 1) & (dot < 0), (i == 0) & (dot > 0)
        side = (i == self.n[0] - 1) & ((d[:, 0] * self.cpm[j] + d[:, 1] * self.spm[j]) < 0)
        ends = ((k == 0) & (d[:, 2] > 0)) | ((k == self.n[2] - 1) & (d[:, 2] < 0))
        return side | ends, torch.zeros_like(side)

    def _roots(self, A, B, C):
        disc = B * B - A * C
        s = torch.sqrt(disc.clamp(min=0.0))
        q = torch.where(B >= 0, -(B + s), s - B)
        r1, r2 = q / A, C / q
        ok = disc > 0
        return torch.where(ok, torch.minimum(r1, r2), INF), torch.where(ok, torch.maximum(r1, r2), INF)

    def _after(self, r, t):
        return torch.where(r > t, r, INF)

    def _cone(self, j, p, d, inv, t):
        c = self.ct[j]
        flat = c.abs() < 1e-12
        cc = c * c
        A, B, C = d[:, 2] * d[:, 2] - cc * inv[0], inv[3] - cc * inv[1], inv[4] - cc * inv[2]
        lo, hi = self._roots(A, B, C)
        same = lo == hi
        lin = -(C / (2.0 * B))
        lo = torch.where(A == 0, torch.where(B == 0, INF, lin), torch.where(same, INF, lo))
        hi = torch.where((A == 0) | same, INF, hi)

        def own(r):
            z = p[2] + r * d[:, 2]
            return torch.where(torch.where(c > 0, z > 0, z < 0), r, INF)
        cand = torch.minimum(self._after(own(lo), t), self._after(own(hi), t))
        plane = torch.where(d[:, 2] != 0, -(p[2] / d[:, 2]), INF)
        return torch.where(flat, self._after(plane, t), cand)

    def _half(self, k, p, d, t):
        c, s = self.cp[k], self.sp[k]
        den = c * d[:, 1] - s * d[:, 0]
        r = -((c * p[1] - s * p[0]) / den)
        h = c * (p[0] + r * d[:, 0]) + s * (p[1] + r * d[:, 1])
        return torch.where((den != 0) & (h > 0), self._after(r, t), INF)

    def walk(self, v, d, lengths):
        """Cells met from the centre of voxel v along d: list of (voxel or -1, t_in, t_out, after a hole) per
        step (only the voxels unless `lengths`), and whether the line ended at the core."""
        sph = self.coord == I.SPHERICAL
        n1, n2, n3 = self.n
        p = self.centre(v)
        i, j, k = self.ijk(v)
        dx, dy, dz = d[:, 0], d[:, 1], d[:, 2]
        xy = (dx * dx + dy * dy, p[0] * dx + p[1] * dy, p[0] * p[0] + p[1] * p[1])
        inv = (xy[0] + dz * dz, xy[1] + p[2] * dz, xy[2] + p[2] * p[2]) if sph else xy
        inv = inv + (p[2] * dz, p[2] * p[2])
        t = torch.zeros_like(dx)
        live = torch.ones_like(dx, dtype=torch.bool)
        hole = torch.zeros_like(live)
        core = torch.zeros_like(live)
        out = []

        def shell(m):
            r = self.e[0][m]
            lo, hi = self._roots(inv[0], inv[1], inv[2] - r * r)
            on = inv[0] > 0
            return torch.where(on, lo, INF), torch.where(on, hi, INF)
        for _ in range(4 * (n1 + n2 + n3) + 16):
            if not bool(live.any()):
                break
            c = [None] * 6
            lo, hi = shell(i)
            c[0] = torch.where(lo < hi, self._after(lo, t), INF)
            c[1] = self._after(shell(i + 1)[1], t)
            if sph:
                c[2] = torch.where(j >= 1, self._cone(j, p, d, inv, t), INF)
                c[3] = torch.where(j + 1 <= n2 - 1, self._cone(j + 1, p, d, inv, t), INF)
                c[4] = self._half(k, p, d, t)
                c[5] = self._half((k + 1) % n3, p, d, t)
            else:
                c[2] = self._half(j, p, d, t)
                c[3] = self._half((j + 1) % n2, p, d, t)
                c[4] = torch.where(dz < 0, self._after((self.e[2][k] - p[2]) / dz, t), INF)
                c[5] = torch.where(dz > 0, self._after((self.e[2][k + 1] - p[2]) / dz, t), INF)
            best = torch.stack(c).amin(0)
            live = live & torch.isfinite(best)
            cell = torch.where(live, (i * n2 + j) * n3 + k, -1).int()
            out.append((cell, t, best, hole) if lengths else cell)
            hit = [q == best for q in c]
            leave = hit[1] & (i == n1 - 1)
            at_core = hit[0] & (i == 0)
            i = (i - (hit[0] & (i > 0)).long() + (hit[1] & (i < n1 - 1)).long())
            if sph:
                j = j - hit[2].long() + hit[3].long()
                k = (k - hit[4].long() + hit[5].long()) % n3
            else:
                leave = leave | (hit[4] & (k == 0)) | (hit[5] & (k == n3 - 1))
                j = (j - hit[2].long() + hit[3].long()) % n2
                k = (k - hit[4].long() + hit[5].long()).clamp(0, n3 - 1)
            at_core = at_core & ~leave
            t = best
            hole = torch.zeros_like(live)
            if sph:
                core = core | (live & at_core)
                live = live & ~leave & ~at_core
            else:  # across the hole to the far side of its surface, or out through an end plane
                far = shell(torch.zeros_like(i))[1]
                tz = torch.where(dz > 0, (self.e[2][n3] - p[2]) / dz, torch.where(dz < 0, (self.e[2][0] - p[2]) / dz, INF))
                live = live & ~leave & ~(at_core & (tz <= far))
                hole = live & at_core
                if bool(hole.any()):
                    q = hole.nonzero()[:, 0]
                    x, y, z = (p[a][q] + far[q] * d[q, a] for a in range(3))
                    g = self.cp[:, None] * y - self.sp[:, None] * x
                    inside = (g >= 0) & (torch.roll(g, -1, 0) < 0)
                    j = j.clone()
                    k = k.clone()
                    j[q] = inside.int().argmax(0)
                    k[q] = (z[None] >= self.e[2][1:-1, None]).sum(0)
                    i = torch.where(hole, 0, i)
                    t = torch.where(hole, far, t)
        return out, core


class _Model:
    """Characteristics of a grid and formal solutions along them."""

    def __init__(self, coord, edges, dirs, wts, dev):
        self.lines = L = _Lines(coord, edges, dev)
        self.nv, self.na, self.dev = L.n[0] * L.n[1] * L.n[2], len(wts), dev
        self.sph = coord == I.SPHERICAL
        d = torch.tensor(dirs, device=dev)
        self.dirs, self.wts = d, torch.tensor(wts, device=dev)
        v = torch.arange(self.nv, device=dev).repeat(self.na)
        w = torch.arange(self.na, device=dev).repeat_interleave(self.nv)
        dd = d[w]
        cells = torch.stack(L.walk(v, -dd, False)[0] + L.walk(v, dd, False)[0])  # steps x lines
        enter, leave = L.starts(v, dd)
        first = (enter | leave).view(self.na, self.nv)
        hit = torch.zeros((self.na, self.nv + 1), dtype=torch.bool, device=dev)
        cells = torch.where(cells < 0, self.nv, cells).view(-1, self.na, self.nv)
        for a in range(self.na):
            hit[a, cells[:, a, first[a]].reshape(-1).long()] = True
        chosen = first.clone()
        per = cells.permute(2, 1, 0).long().contiguous()  # voxel, angle, step
        for u in range(self.nv):  # then one through every voxel not hit yet, in voxel order
            need = ~hit[:, u]
            chosen[:, u] |= need
            hit.scatter_(1, torch.where(need[:, None], per[u], self.nv), True)
        del cells, per
        w, v = chosen.nonzero(as_tuple=True)
        back, core = L.walk(v, -d[w], True)
        fwd, _ = L.walk(v, d[w], True)
        vox, ln, rest = [], [], []
        for q in range(len(back) - 1, 0, -1):  # the upstream half, reversed
            c, t0, t1, _ = back[q]
            vox.append(c)
            ln.append(t1 - t0)
            # the cell before this one downstream lies across a hole when that step began after one
            rest.append(back[q + 1][3] & (back[q + 1][0] >= 0) if q + 1 < len(back) else torch.zeros_like(core))
        r0 = back[1][3] & (back[1][0] >= 0) if len(back) > 1 else torch.zeros_like(core)
        vox.append(fwd[0][0])
        ln.append(back[0][2] + fwd[0][2])
        rest.append(r0)
        for c, t0, t1, h in fwd[1:]:
            vox.append(c)
            ln.append(t1 - t0)
            rest.append(h)
        vox, rest = torch.stack(vox), torch.stack(rest)  # steps x characteristics
        ok = vox >= 0
        first_at = ok.int().argmax(0)
        K, R = vox.shape
        row = torch.arange(K, device=dev)[:, None]
        self.start = row == first_at[None]
        self.ok, self.vox, self.len = ok, vox.clamp(min=0).long(), torch.where(ok, torch.stack(ln), 0.0)
        self.run0 = ok & (self.start | rest)
        self.core = core
        self.v1 = self.vox.gather(0, first_at[None])[0]
        self.w = w
        key = (w[None] * self.nv + self.vox)
        tot = torch.zeros(self.na * self.nv, dtype=torch.float64, device=dev).index_add_(0, key[ok], self.len[ok])
        self.c = torch.where(ok, self.len * (self.wts[w][None] / tot[key]), 0.0)  # gather weight of a segment
        nxt = torch.zeros_like(ok)
        nxt[:-1] = ok[1:] & ~self.run0[1:]
        self.more = ok & nxt  # the run goes on behind this segment

    def at(self, field):
        return field.index_select(0, self.vox.reshape(-1)).view(self.vox.shape)

    def weights(self, chi):
        x = torch.where(self.ok, self.at(chi) * self.len, 1.0)
        p = torch.ones_like(x)
        p = torch.cat((x[1:], p[-1:]))
        para = self.more & (p.detach() >= 0.5 * x.detach())
        p = torch.where(para, p, 1.0)
        e0 = -torch.expm1(-x)
        big = x.detach() >= 0.5
        xs, xb = torch.where(big, 0.25, x), torch.where(big, x, 1.0)
        # f1 = (x - e0) / x and f2 = (x (x - e0) - (x^2 - 2 (x - e0))) / x; for small x by their power series
        h1 = torch.zeros_like(x)
        h2 = torch.zeros_like(x)
        for m in range(22, 1, -1):
            h1 = 1.0 / math.factorial(m) - xs * h1
            if m >= 3:
                h2 = (m - 2) / math.factorial(m) - xs * h2
        eb = -torch.expm1(-xb)
        f1 = torch.where(big, (xb - eb) / xb, xs * h1)
        f2 = torch.where(big, (xb * (xb - eb) - (xb * xb - 2.0 * (xb - eb))) / xb, xs * xs * h2)
        al = e0 - f1 - torch.where(para, f2 / (x + p), 0.0)
        be = f1 + torch.where(para, f2 / p, 0.0)
        ga = torch.where(para, -x * f2 / (p * (x + p)), 0.0)
        return torch.exp(-x), al, be, ga

    def solution(self, S, chi, B, lam=False, flux=False, wts=None):
        """J (with Lambda* and the flux in the local basis if asked for); wts: weights(chi), if in hand."""
        E, al, be, ga = self.weights(chi) if wts is None else wts
        Sv = self.at(S)
        Sm = torch.where(self.run0, Sv, torch.cat((Sv[:1], Sv[:-1])))
        Sp = torch.cat((Sv[1:], Sv[-1:]))
        src = al * Sm + be * Sv + ga * Sp
        cur = torch.where(self.core, B[self.v1], 0.0) if B is not None else torch.zeros_like(src[0])
        rows = []
        for e, b in zip(torch.where(self.ok, E, 1.0).unbind(0), torch.where(self.ok, src, 0.0).unbind(0)):
            cur = torch.addcmul(b, e, cur)
            rows.append(cur)
        val = self.c * torch.stack(rows)
        J = torch.zeros(self.nv, dtype=torch.float64, device=self.dev).index_add(0, self.vox.reshape(-1), val.reshape(-1))
        out = [J]
        if lam:
            gm = torch.cat((torch.zeros_like(ga[:1]), ga[:-1]))
            l = self.c * (be + torch.where(self.run0, al, gm * E))
            out.append(torch.zeros_like(J).index_add(0, self.vox.reshape(-1), l.reshape(-1)))
        if flux:
            i, j, k = self.lines.ijk(torch.arange(self.nv, device=self.dev))
            G = self.lines
            C = [torch.zeros_like(J).index_add(0, self.vox.reshape(-1), (val * self.dirs[self.w, a]).reshape(-1)) for a in range(3)]
            if self.sph:
                st, ct, cp, sp = G.stm[j], G.ctm[j], G.cpm[k], G.spm[k]
                basis = ((st * cp, st * sp, ct), (ct * cp, ct * sp, -st), (-sp, cp, torch.zeros_like(cp)))
            else:
                cp, sp, o = G.cpm[j], G.spm[j], torch.zeros_like(C[0])
                basis = ((cp, sp, o), (-sp, cp, o), (o, o, o + 1.0))
            out.append(torch.stack([4.0 * math.pi * sum(b * c for b, c in zip(row, C)) for row in basis], 1))
        return out if len(out) > 1 else J


def _ng(y):
    """Order-2 Ng step from four iterates, newest first; the newest one where the system is singular."""
    W = 1.0 / (y[0] * y[0])
    r = [y[q] - y[q + 1] for q in range(3)]
    d1, d2 = r[0] - r[1], r[0] - r[2]
    a, b, c = (W * d1 * d1).sum(), (W * d1 * d2).sum(), (W * d2 * d2).sum()
    u, v = (W * d1 * r[0]).sum(), (W * d2 * r[0]).sum()
    det = a * c - b * b
    if not abs(float(det)) > 1e-14 * float(a * c):
        return None
    p, q = (u * c - v * b) / det, (a * v - b * u) / det
    return (1.0 - p - q) * y[0] + p * y[1] + q * y[2]


def _ali(fs, L, S, eps, B, steps, ng):
    hist, J = [], None
    for _ in range(steps):
        J = fs(S)
        S = S + ((1.0 - eps) * J + eps * B - S) / (1.0 - (1.0 - eps) * L)
        hist.insert(0, S)
        hist = hist[:4]
        if ng and len(hist) == 4:
            new = _ng(hist)
            if new is not None:
                S, hist = new, []
    return S, J


def _bicgstab(op, b, D, limit):
    """x of op(x) = b with the diagonal D as its preconditioner; None if it is not found within `limit` seconds."""
    began = time.monotonic()
    x = b / D
    r = b - op(x)
    r0 = r.clone()
    rho = al = om = torch.ones((), dtype=b.dtype, device=b.device)
    v = p = torch.zeros_like(b)
    best, still = INF, 0
    for _ in range(4000):
        size = float((r / D).abs().max() / x.abs().max())
        if size < 3e-14 or still > 10:
            break
        best, still = (size, 0) if size < 0.9 * best else (best, still + 1)
        if time.monotonic() - began > limit:
            return None
        new = (r0 * r).sum()
        p = r + (new / rho) * (al / om) * (p - om * v)
        rho = new
        ph = p / D
        v = op(ph)
        al = rho / (r0 * v).sum()
        s = r - al * v
        sh = s / D
        t = op(sh)
        om = (t * s).sum() / (t * t).sum()
        x = x + al * ph + om * sh
        r = s - om * t
    return x if best < 1e-11 else None


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    lines = max(n[0] * n[1] * n[2] for n in _shapes(case)) * case["mu"] * case["phi"]
    if lines > (1.3e6 if dev == "cuda" else 1e5) or (kind == "line" and case["lstar"] == rt.RT_LSTAR_NN):
        return None  # takes too long (or: the iterates depend on an operator of the library's own)
    x = _inputs(case, seed)
    dirs, wts = I.angle_set(case["mu"], case["phi"])
    models = [_Model(case["coord"], _edges(case["coord"], n), dirs, wts, dev) for n in _shapes(case)]
    M = models[0]
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    fields = [tuple(t(a) for a in m) for m in x["members"]]
    chi, eps, B = fields[0]
    if kind in ("fs", "sweep"):
        J, L, F = M.solution(B, chi, B, True, True)
        return dict(J=J, L=L, F=F) if kind == "fs" else dict(J=J, F=F)
    if kind in ("ali", "batch"):
        res = {}
        for m, (chi, eps, B) in enumerate(fields):
            M = models[m % len(models)]
            wt = M.weights(chi)
            L = M.solution(B, chi, B, True, wts=wt)[1]
            S, J = _ali(lambda s: M.solution(s, chi, B, wts=wt), L, B, eps, B, case["steps"], kind == "ali")
            res.update({"S%d" % m: S, "J%d" % m: J} if kind == "batch" else dict(S=S, J=J))
        return res
    if kind == "line":
        phi, wq = I.line_profile(case["members"])
        chi_c, chi_l = t(x["chi_c"]), t(x["chi_l"])
        ks = [chi_c + chi_l * f for f in phi]
        wt = [M.weights(c) for c in ks]
        src = lambda k, s: (chi_c * B + chi_l * phi[k] * s) / ks[k]  # noqa: E731
        L = sum(wq[k] * phi[k] * (chi_l * phi[k] / ks[k]) * M.solution(B, ks[k], B, True, wts=wt[k])[1]
                for k in range(len(phi)))
        fs = lambda s: sum(wq[k] * phi[k] * M.solution(src(k, s), ks[k], B, wts=wt[k]) for k in range(len(phi)))  # noqa: E731
        S, J = _ali(fs, L, B, eps, B, case["steps"], True)
        return dict(S=S, J=J)
    wt = M.weights(chi)
    J0, L = M.solution(torch.zeros_like(B), chi, B, True, wts=wt)
    S = _bicgstab(lambda s: s - (1.0 - eps) * M.solution(s, chi, None, wts=wt), (1.0 - eps) * J0 + eps * B,
                  1.0 - (1.0 - eps) * L, 10.0)
    if S is None:
        return None
    if kind == "solve":
        return dict(S=S, J=M.solution(S, chi, B, wts=wt))
    s, c, b = (q.clone().requires_grad_(True) for q in (S, chi, B))
    J, F = M.solution(s, c, b, flux=True)
    gS, gJ, gF = (t(g) for g in x["g"])
    back = lambda u, f, wrt: torch.autograd.grad((J, F), wrt, (u, f), retain_graph=True)  # noqa: E731
    rhs = gS + back(gJ, gF, s)[0]
    zero = torch.zeros_like(gF)
    lam = _bicgstab(lambda u: u - back((1.0 - eps) * u, zero, s)[0], rhs, 1.0 - (1.0 - eps) * L, 10.0)
    if lam is None:
        return None
    dchi, dB = back(gJ + (1.0 - eps) * lam, gF, (c, b))
    # the flux that comes back is that of the iteration's first formal solution, from S = B (later ones leave it)
    F0 = M.solution(B, chi, B, flux=True)[1]
    return dict(S=S, J=J.detach(), F=F0, dchi=dchi, deps=lam * (B - J.detach()), dB=dB + eps * lam)
