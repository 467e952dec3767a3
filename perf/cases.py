"""Timed cases: the calls a user of the library makes, over the sizes it is used at.

Geometries are generated here (bars, bond-wire arrays, stacked plates; jittered
meshes of the shapes and panel sizes of the bench workloads), a case's plan is
what a program keeps between calls, and its currents come from the seed.  The
right-hand sides of a product are frequencies x ports, or the Krylov vectors of
as many solves: from one (one port at one frequency) to 128 (8 ports at 16
frequencies).

exact() evaluates the same operator in 64 bits with plain numpy and torch: the
loop matrix as a sparse matrix, the projection and near blocks as the plan
exports them, the grid convolution by torch.fft on a table of 1/R.
"""
import math

import numpy as np
import torch

from paper_2210_04891_gb300 import (PREC_DF, PREC_FP64, PREC_MIXED, REFINE_DF, SPACE_BRANCH, SPACE_LOOP, api, native)

UM = 1e-6
MU0 = 4e-7 * math.pi
PREC = {"fp64": PREC_FP64, "mixed": PREC_MIXED, "df": PREC_DF}
SPACE = {"loop": SPACE_LOOP, "branch": SPACE_BRANCH}


def listed():
    return [
        # The smallest call: one product of a straight interconnect (1.5k triangles) with one vector in
        # the default precision, as a user's own iterative solver makes it.
        dict(name="bar_matvec_fp64_r1", op="matvec", shape="bar", n=125, prec="fp64", space="loop", rhs=1),
        # A whole port solve of that interconnect at one frequency, mixed precision refined to 1e-6.
        dict(name="bar_solve_df", op="solve", shape="bar", n=125, freqs=1),
        # A few ports of a medium wire array at one frequency: an odd, small number of vectors.
        dict(name="wires_matvec_mixed_r3", op="matvec", shape="wires", n=3, seg=124, prec="mixed", space="loop",
             rhs=3),
        # The default precision on the same class of array, eight ports at one frequency.
        dict(name="wires_matvec_fp64_r8", op="matvec", shape="wires", n=8, seg=77, prec="fp64", space="loop", rhs=8),
        # The full wire array (40k triangles) at every port and frequency: the Arnoldi product of its solve.
        dict(name="wires_matvec_mixed_r128", op="matvec", shape="wires", n=8, seg=156, lo=32, prec="mixed",
             space="loop", rhs=128),
        # The default precision at a frequency sweep's width: the plain solve's product.
        dict(name="wires_matvec_fp64_r48", op="matvec", shape="wires", n=8, seg=156, lo=32, prec="fp64",
             space="loop", rhs=48),
        # The residual product of a refined solve (double-float), one port per wire at two frequencies.
        dict(name="wires_matvec_df_r16", op="matvec", shape="wires", n=8, seg=156, lo=32, prec="df",
             space="loop", rhs=16),
        # The preconditioner of the full array's solve, once per Arnoldi step.
        dict(name="wires_precond_mixed_r128", op="precond", shape="wires", n=8, seg=156, lo=32, prec="mixed",
             rhs=128),
        # Two stacked plates: branch voltages of branch currents (what post-processing asks for), a wide grid.
        dict(name="plates_matvec_mixed_r32", op="matvec", shape="plates", n=100, prec="mixed", space="branch",
             rhs=32),
        # The plates' preconditioner: a wide band instead of the wires' narrow one.
        dict(name="plates_precond_mixed_r4", op="precond", shape="plates", n=56, prec="mixed", rhs=4),
        # The grid convolution alone, on the plane pair's grid (its (y, z) plane does not fit one CTA).
        dict(name="convolve_mixed_256x256x32", op="convolve", gx=256, gy=256, gz=32, prec="mixed", rhs=24),
        # Uneven traces stepped together in one call, 32 frequencies each.
        dict(name="batch_matvec_mixed_r32", op="batch", shape="bar", n=500, count=6, prec="mixed", rhs=32),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["matvec", "matvec", "matvec", "matvec", "precond", "convolve", "solve", "batch"])
    if op == "convolve":
        gx, gy, gz = (2 ** rng.randint(3, 8), 2 ** rng.randint(3, 8), 2 ** rng.randint(3, 5))
        most = max(1, min(96, 24 * 256 * 256 * 32 // (gx * gy * gz)))
        prec = rng.choice(["mixed", "mixed", "fp64"])
        most = max(1, most // (8 if prec == "fp64" else 1))
        return dict(op=op, gx=gx, gy=gy, gz=gz, prec=prec, rhs=_logint(rng, 1, most))
    if op == "solve":
        return dict(op=op, shape="bar", n=_logint(rng, 20, 180), freqs=rng.randint(1, 4))
    if op == "batch":
        return dict(op=op, shape="bar", n=_logint(rng, 100, 500), count=rng.randint(2, 6), prec="mixed",
                    rhs=_logint(rng, 1, 32))
    prec = rng.choice(["mixed", "fp64", "df"]) if op == "matvec" else rng.choice(["mixed", "mixed", "fp64"])
    rhs = _logint(rng, 1, {"mixed": 128, "fp64": 40, "df": 64}[prec])
    shape = rng.choice(["bar", "wires", "plates"])
    c = dict(op=op, shape=shape, prec=prec, rhs=rhs)
    if op == "matvec":
        c["space"] = rng.choice(["loop", "loop", "branch"])
    if shape == "bar":
        c["n"] = _logint(rng, 20, 600)
    elif shape == "wires":
        c["n"], c["seg"], c["lo"] = rng.randint(1, 8), _logint(rng, 20, 150), rng.choice([8, 16, 32])
    else:
        c["n"] = _logint(rng, 16, 90 if op == "matvec" else 56)
    return c


# ---------------------------------------------------------------- geometry

def _box(nx, ny, nz, hx, hy, hz, origin, jitter, rng):
    """Closed surface of a box of nx x ny x nz cells, each quad cut along alternating diagonals; vertices
    inside a face move in its plane by up to jitter cells.  (xyz, triangles, source faces, sink faces.)"""
    dims = (nx, ny, nz)

    def code(p):
        return (p[..., 0] * (ny + 1) + p[..., 1]) * (nz + 1) + p[..., 2]

    tris, tags = [], []
    for axis in range(3):
        ua, wa = [a for a in range(3) if a != axis]
        u, w = (v.ravel() for v in np.meshgrid(np.arange(dims[ua]), np.arange(dims[wa]), indexing="ij"))
        for side in (0, 1):
            q = []
            for du, dw in ((0, 0), (1, 0), (1, 1), (0, 1)):
                p = np.empty((u.size, 3), np.int64)
                p[:, axis], p[:, ua], p[:, wa] = side * dims[axis], u + du, w + dw
                q.append(code(p))
            a, b, c, d = q
            # (u, w) x normal is right-handed for axes 0 and 2: keep the outward normal on the right
            if (side == 1) != (axis != 1):
                b, d = d, b
            even = ((u + w) % 2 == 0)[:, None]
            t0 = np.where(even, np.stack([a, b, c], 1), np.stack([a, b, d], 1))
            t1 = np.where(even, np.stack([a, c, d], 1), np.stack([b, c, d], 1))
            tris.append(np.stack([t0, t1], 1).reshape(-1, 3))
            tags.append(np.full(2 * u.size, 2 * axis + side))
    tri, tag = np.concatenate(tris), np.concatenate(tags)
    used, inv = np.unique(tri.ravel(), return_inverse=True)
    tri = inv.reshape(tri.shape)
    ijk = np.stack([used // ((ny + 1) * (nz + 1)), used // (nz + 1) % (ny + 1), used % (nz + 1)], 1)
    h = np.array([hx, hy, hz])
    on = (ijk == 0) | (ijk == np.array(dims))
    move = rng.uniform(-jitter, jitter, ijk.shape) * ((on.sum(1) == 1)[:, None] & ~on)
    xyz = (ijk + move) * h + np.asarray(origin)
    return xyz, tri, np.nonzero(tag == 0)[0], np.nonzero(tag == 1)[0]


def _wire(seg, sides, radius, seg_len, y0, jitter, rng):
    """Closed round wire along x (a sides-gon of seg rings, fan caps)."""
    x = np.arange(seg + 1) * seg_len
    x[1:-1] += rng.uniform(-jitter, jitter, seg - 1) * seg_len
    th = 2 * np.pi * np.arange(sides) / sides
    ring = np.stack([np.repeat(x, sides), np.tile(y0 + radius * np.cos(th), seg + 1),
                     np.tile(radius * np.sin(th), seg + 1)], 1)
    xyz = np.concatenate([ring, [[x[0], y0, 0.0], [x[-1], y0, 0.0]]])
    s, k = (v.ravel() for v in np.meshgrid(np.arange(seg), np.arange(sides), indexing="ij"))
    k1 = (k + 1) % sides
    a, b, c, d = s * sides + k, s * sides + k1, (s + 1) * sides + k1, (s + 1) * sides + k   # outward on the right
    even = ((s + k) % 2 == 0)[:, None]
    t0 = np.where(even, np.stack([a, b, c], 1), np.stack([a, b, d], 1))
    t1 = np.where(even, np.stack([a, c, d], 1), np.stack([b, c, d], 1))
    r, r1 = np.arange(sides), (np.arange(sides) + 1) % sides
    c0, c1 = ring.shape[0], ring.shape[0] + 1
    cap0 = np.stack([np.full(sides, c0), r1, r], 1)
    cap1 = np.stack([np.full(sides, c1), seg * sides + r, seg * sides + r1], 1)
    n = 2 * s.size
    tri = np.concatenate([np.stack([t0, t1], 1).reshape(-1, 3), cap0, cap1])
    return xyz, tri, n + r, n + sides + r


def _mesh(case):
    """(xyz, triangles, conductor of each, conductivities, ports, panel size) of a case's geometry."""
    rng = np.random.default_rng(11)
    parts, sigma, cell = [], 5.8e7, 0.0
    if case["shape"] == "bar":          # 20 x 10 um copper trace, 8 um panels
        parts.append(_box(case["n"], 2, 1, 8 * UM, 10 * UM, 10 * UM, (0, 0, 0), 0.15, rng))
        cell = 16 * UM
    elif case["shape"] == "wires":      # 25 um gold bond wires at 100 um pitch
        sigma, cell = 4.1e7, 16 * UM
        for w in range(case["n"]):
            parts.append(_wire(case["seg"], 16, 12.5 * UM, 12.8 * UM, w * 100 * UM, 0.1, rng))
    else:                               # two 35 um copper plates 100 um apart, 40 um panels
        cell = 40 * UM
        for k in range(2):
            parts.append(_box(case["n"], case["n"], 1, 40 * UM, 40 * UM, 35 * UM, (0, 0, k * 135 * UM), 0.15, rng))
    xyz, tri, cond, ports, nv, nt = [], [], [], [], 0, 0
    for i, (x, t, src, snk) in enumerate(parts):
        xyz.append(x)
        tri.append(t + nv)
        cond.append(np.full(len(t), i))
        ports.append((src + nt, snk + nt))
        nv, nt = nv + len(x), nt + len(t)
    return (np.concatenate(xyz), np.concatenate(tri).astype(np.int32), np.concatenate(cond).astype(np.int32),
            np.full(len(parts), sigma), ports, cell)


def _grid(xyz, cell, lo=8):
    """Nodes per axis: the power of two that covers the extent at the given spacing, lo to 256."""
    out = []
    for e in xyz.max(0) - xyz.min(0):
        n = lo
        while n < 256 and (n - 1) * cell < e:
            n *= 2
        out.append(n)
    return tuple(out)


def _plan(case):
    xyz, tri, cond, sigma, ports, cell = _mesh(case)
    mesh = api.Mesh(xyz, tri, cond, sigma)
    loops = api.Loops(mesh, ports)
    grid = _grid(xyz, cell, case.get("lo", 8))
    return api.Plan(mesh, loops, dict(grid=grid, order=3, near_factor=4.0, near_min_diam=2.0, n_touch=8, h0=0.0))


def _omega(rhs, lo=6.0, hi=10.0):
    return 2 * np.pi * np.logspace(lo, hi, rhs) if rhs > 1 else np.array([2 * np.pi * 1e9])


def _currents(rhs, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(rhs, n, dtype=torch.complex128, device="cuda", generator=g)


# ---------------------------------------------------------------- cases

def _part(case, i):
    """Trace i of a batch: uneven lengths, the longest first."""
    return dict(shape=case["shape"], n=max(20, case["n"] * (case["count"] - i) // case["count"]))


def prepare(case, seed):
    s = dict(case=case)
    op = case["op"]
    if op == "convolve":
        # a plan's grid is free of its mesh: a short bar stretched over the grid's box
        xyz, tri, cond, sigma, ports, _ = _mesh(dict(shape="bar", n=20))
        mesh = api.Mesh(xyz, tri, cond, sigma)
        loops = api.Loops(mesh, ports)
        s["plan"] = api.Plan(mesh, loops, dict(grid=(case["gx"], case["gy"], case["gz"])))
        dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
        g = torch.Generator(device="cuda").manual_seed(seed)
        s["x"] = torch.randn(case["rhs"], case["gx"], case["gy"], case["gz"], dtype=dt, device="cuda", generator=g)
        return s
    if op == "batch":
        s["plans"] = [_plan(_part(case, i)) for i in range(case["count"])]
        s["batch"] = api.Batch(s["plans"])
        s["x"] = [_currents(case["rhs"], p.nl, seed + i) for i, p in enumerate(s["plans"])]
        s["y"] = [torch.empty_like(x) for x in s["x"]]
        s["omega"] = [_omega(case["rhs"], 7.0, 9.7)] * case["count"]
        return s
    plan = s["plan"] = _plan(case)
    if op == "solve":
        # a sweep whose frequencies are the caller's own
        f = np.random.default_rng(seed).uniform(0.9, 1.1, case["freqs"])
        s["freqs"] = f * np.logspace(8.5, 9.5, case["freqs"])
        return s
    s["omega"] = _omega(case["rhs"])
    n = plan.nb if case.get("space") == "branch" else plan.nl
    s["x"] = _currents(case["rhs"], n, seed)
    if op == "precond":
        # 16 frequencies at most: the right-hand sides of one frequency are its ports
        nf = min(16, case["rhs"])
        s["omega"] = np.repeat(_omega(nf), -(-case["rhs"] // nf))[:case["rhs"]]
        s["out"] = torch.empty_like(s["x"])
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "matvec":
        return api.pfft_matvec(s["plan"], s["x"], s["omega"], SPACE[c["space"]], PREC[c["prec"]])
    if op == "precond":
        return api.pfft_precond_apply(s["plan"], s["x"], s["omega"], out=s["out"], prec=PREC[c["prec"]])
    if op == "convolve":
        return api.pfft_convolve(s["plan"], s["x"].clone(), PREC[c["prec"]])   # the call is in place
    if op == "batch":
        return s["batch"].matvec(s["x"], s["omega"], SPACE_LOOP, PREC[c["prec"]], graph=True, outs=s["y"])
    return api.sie_solve(s["plan"], s["freqs"], tol=1e-6, prec=PREC_MIXED, refine=REFINE_DF)[0]


# ---------------------------------------------------------------- work

def _counts(case):
    """Triangles, loops, branches, near pairs per triangle and grid nodes of a geometry, from its numbers."""
    n = case["n"]
    if case["shape"] == "bar":
        nt, parts, near = 4 * (2 * n + n + 2), 1, 190
    elif case["shape"] == "wires":
        nt, parts, near = n * 32 * (case["seg"] + 1), n, 270
    else:
        nt, parts, near = 2 * (4 * n * n + 8 * n), 2, 180
    xyz, _, _, _, _, cell = _mesh(case)
    gx, gy, gz = _grid(xyz, cell, case.get("lo", 8))
    return nt, nt // 2 + 2 * parts, 3 * nt // 2, min(near, nt), gx * gy * gz


def _matvec_work(case, rhs, prec, space):
    nt, nl, nb, near, ng = _counts(case)
    n = nb if space == "branch" else nl
    real, cplx = (4, 8) if prec == "mixed" else (8, 16)
    # in and out vectors; each near and projection block once; the grids' padded spectrum once
    by = 2 * rhs * n * 16 + nt * (near + 60) * (9 * real + 4) + rhs * 3 * 2 * ng * cplx
    fl = rhs * (36 * nt * (near + 2 * 60) + 3 * 2 * 5 * 8 * ng * math.log2(8 * ng))
    return by, fl


def work(case):
    op = case["op"]
    if op == "convolve":
        ng = case["gx"] * case["gy"] * case["gz"]
        c = 16 if case["prec"] == "fp64" else 8
        return dict(bytes=2 * case["rhs"] * ng * c, flops=case["rhs"] * 2 * 5 * 8 * ng * math.log2(8 * ng))
    if op == "matvec":
        by, fl = _matvec_work(case, case["rhs"], case["prec"], case["space"])
        return dict(bytes=by, flops=fl)
    if op == "batch":
        w = [_matvec_work(_part(case, i), case["rhs"], case["prec"], "loop") for i in range(case["count"])]
        return dict(bytes=sum(v[0] for v in w), flops=sum(v[1] for v in w))
    nt, nl, nb, near, ng = _counts(case)
    if op == "precond":
        # vectors in and out, the factor of each frequency once
        band = {"bar": 12, "wires": 33, "plates": 4 * case["n"]}[case["shape"]]
        c = 8 if case["prec"] == "mixed" else 16
        nf = min(16, case["rhs"])
        return dict(bytes=2 * case["rhs"] * nl * 16 + nf * nt * band * c, flops=case["rhs"] * 16 * nt * band)
    by, fl = _matvec_work(case, case["freqs"], "mixed", "loop")
    return dict(bytes=9 * by, flops=9 * fl)   # about nine iterations


# ---------------------------------------------------------------- 64-bit values

class _Exact:
    """The operator of a plan in complex128 with torch: see the module's text."""

    def __init__(self, case):
        xyz, tri, cond, sigma, ports, _ = _mesh(case)
        plan = self.plan = _plan(case)
        dev = self.dev = torch.device("cuda")
        self.nt, self.nb, self.nl, self.np = len(tri), plan.nb, plan.nl, plan.np
        self.sigma, self.cond, self.grid = sigma, cond, plan.params["grid"]
        # geometry: Gram blocks int (r - v_k).(r - v_l) dS / (4 A^2) and the local edges of each branch
        p = xyz[tri]
        area = 0.5 * np.linalg.norm(np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), axis=1)
        c = p.mean(1)
        quad = (np.einsum("tij,tij->t", p, p) + 9 * np.einsum("ti,ti->t", c, c)) / 12
        pc = np.einsum("tki,ti->tk", p, c)
        gram = (quad[:, None, None] - pc[:, :, None] - pc[:, None, :] + np.einsum("tki,tli->tkl", p, p))
        self.gram = gram / (4 * area[:, None, None])
        row_ptr, col, val, br = plan.loops.export()
        far = ~(tri[br][:, :, :, None] == tri[br][:, ::-1, None, :]).any(-1)   # [nb, 2, 3]: vertex not shared
        self.br, self.loc = br, far.argmax(-1)
        self.tb = np.full((self.nt, 3), -1)
        self.ts = np.zeros((self.nt, 3))
        for side, sign in ((0, 1.0), (1, -1.0)):
            self.tb[br[:, side], self.loc[:, side]] = np.arange(self.nb)
            self.ts[br[:, side], self.loc[:, side]] = sign
        rows = np.repeat(np.arange(self.nl), np.diff(row_ptr))
        self.A = self._sparse(rows, col, val.astype(np.float64), (self.nl, self.nb + self.np))
        self.At = self._sparse(col, rows, val.astype(np.float64), (self.nb + self.np, self.nl))
        # near field and projection as sparse matrices over (triangle, edge)
        ptr, ncol = plan.export(native.EXPORT_NEAR_PTR), plan.export(native.EXPORT_NEAR_COL)
        self.near = self._blocks(np.repeat(np.arange(self.nt), np.diff(ptr)), ncol, plan.export(native.EXPORT_LD),
                                 (3, 1), (3, 1), (3 * self.nt, 3 * self.nt))
        pp, pn = plan.export(native.EXPORT_PROJ_PTR), plan.export(native.EXPORT_PROJ_NODE)
        W = plan.export(native.EXPORT_PROJ_W)
        t = np.repeat(np.arange(self.nt), np.diff(pp))
        ng = int(np.prod(self.grid))
        self.B = self._blocks(pn, t, W, (1, ng), (3, 1), (3 * ng, 3 * self.nt))
        self.Bt = self._blocks(t, pn, W.transpose(0, 2, 1), (3, 1), (1, ng), (3 * self.nt, 3 * ng))
        self.H = _kernel_spectrum(xyz, self.grid)

    def _sparse(self, r, c, v, shape):
        r, c, v = (a if torch.is_tensor(a) else torch.from_numpy(np.ascontiguousarray(a)) for a in (r, c, v))
        i = torch.stack([r.to(self.dev, torch.int64), c.to(self.dev, torch.int64)])
        return torch.sparse_coo_tensor(i, v.to(self.dev), shape).coalesce().to_sparse_csr()

    def _blocks(self, r, c, b, mr, mc, shape):
        """3 x 3 blocks b[i][k][l] at rows mr[0] r + mr[1] k and columns mc[0] c + mc[1] l."""
        r, c, b = (torch.from_numpy(np.ascontiguousarray(a)).to(self.dev) for a in (r, c, b))
        k = torch.arange(3, device=self.dev)
        rows = (mr[0] * r.long()[:, None, None] + mr[1] * k[:, None]).expand(b.shape)
        cols = (mc[0] * c.long()[:, None, None] + mc[1] * k[None, :]).expand(b.shape)
        return self._sparse(rows.reshape(-1), cols.reshape(-1), b.reshape(-1), shape)

    def zs(self, omega):
        return (1 + 1j) * np.sqrt(omega * MU0 / (2 * self.sigma[self.cond]))

    def product(self, x, omega, space):
        out = [self._product(x[i:i + 16], omega[i:i + 16], space) for i in range(0, x.shape[0], 16)]
        return torch.cat(out)

    def _product(self, x, omega, space):
        R, dev = x.shape[0], self.dev
        a = _apply(self.At, x.T)[:self.nb] if space == "loop" else x.T          # [nb, R]
        tb, ts = torch.from_numpy(self.tb).to(dev), torch.from_numpy(self.ts).to(dev)
        cur = torch.where((tb >= 0)[..., None], a[tb.clamp(min=0)], 0) * ts[..., None]
        flat = cur.reshape(3 * self.nt, R)
        q = _apply(self.B, flat).T.reshape(R * 3, *self.grid)
        phi = _fft_convolve(q, self.H).reshape(R, -1).T
        f = (_apply(self.near, flat) + _apply(self.Bt, phi)).reshape(self.nt, 3, R)
        w = torch.from_numpy(omega).to(dev)
        zs = torch.from_numpy(np.stack([self.zs(o) for o in omega], -1)).to(dev)   # [nt, R]
        ohm = torch.einsum("tkl,tlr->tkr", torch.from_numpy(self.gram).to(dev).to(cur.dtype), cur)
        y = zs[:, None, :] * ohm + 1j * w * MU0 / (4 * math.pi) * f
        br, loc = torch.from_numpy(self.br).long().to(dev), torch.from_numpy(self.loc).to(dev)
        yb = y[br[:, 0], loc[:, 0]] - y[br[:, 1], loc[:, 1]]
        if space == "branch":
            return yb.T.contiguous()
        return _apply(self.A, torch.cat([yb, yb.new_zeros(self.np, R)])).T.contiguous()

    def branch_diagonal(self, omega):
        """Z_b's diagonal: the self and facing terms of each branch's two triangles."""
        ptr, ncol = self.plan.export(native.EXPORT_NEAR_PTR), self.plan.export(native.EXPORT_NEAR_COL)
        L = self.plan.export(native.EXPORT_LDIRECT)
        key = np.repeat(np.arange(self.nt), np.diff(ptr)) * self.nt + ncol
        zs, out = self.zs(omega), np.zeros(self.nb, complex)
        for i in (0, 1):
            t, k = self.br[:, i].astype(np.int64), self.loc[:, i]
            out += zs[t] * self.gram[t, k, k]
            for j in (0, 1):
                u, l = self.br[:, j].astype(np.int64), self.loc[:, j]
                e = np.searchsorted(key, t * self.nt + u)
                out += (1 if i == j else -1) * 1j * omega * MU0 / (4 * math.pi) * L[e, k, l]
        return out


def _apply(S, x):
    """Real sparse times complex dense."""
    v = torch.view_as_real(x.contiguous()).reshape(x.shape[0], -1)
    return torch.view_as_complex((S @ v).reshape(S.shape[0], -1, 2).contiguous())


def _kernel_spectrum(xyz, grid):
    h = (xyz.max(0) - xyz.min(0)) / (np.array(grid) - 1)
    ax = [torch.from_numpy(np.minimum(np.arange(2 * n), 2 * n - np.arange(2 * n)) * s).cuda() for n, s in zip(grid, h)]
    r = torch.sqrt(ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2)
    r[0, 0, 0] = math.inf                       # the kernel's value at zero offset is 0
    return torch.fft.fftn(1.0 / r)


def _fft_convolve(q, H):
    out = torch.empty_like(q)
    s = H.shape
    for i in range(q.shape[0]):
        out[i] = torch.fft.ifftn(torch.fft.fftn(q[i], s=s) * H)[:s[0] // 2, :s[1] // 2, :s[2] // 2]
    return out


def exact(case, seed):
    op = case["op"]
    if op == "convolve":
        s = prepare(case, seed)
        return _fft_convolve(s["x"].to(torch.complex128),
                             _kernel_spectrum(_mesh(dict(shape="bar", n=20))[0], (case["gx"], case["gy"], case["gz"])))
    if op == "batch":
        s = prepare(case, seed)
        return [_Exact(_part(case, i)).product(x, w, "loop") for i, (x, w) in enumerate(zip(s["x"], s["omega"]))]
    s = prepare(case, seed)
    if op == "matvec":
        return _Exact(case).product(s["x"], s["omega"], case["space"])
    nl = s["plan"].nl
    if nl > 6000 or (op == "solve" and nl > 2500):
        return None
    E = _Exact(case)
    if op == "precond":                         # dense solve with P = A diag(Z_b) A^T, one matrix per frequency
        A = E.A.to_dense()[:, :E.nb].to(torch.complex128)
        out = torch.empty_like(s["x"])
        if len(set(s["omega"])) * nl ** 3 > 8e11:
            return None
        for w in sorted(set(s["omega"])):
            P = (A * torch.from_numpy(E.branch_diagonal(w)).cuda()) @ A.T
            at = torch.from_numpy(np.nonzero(s["omega"] == w)[0]).cuda()
            out[at] = torch.linalg.solve(P, s["x"][at].T).T
        return out
    Z = []                                      # the full system's dense solve: Y[q][p] = I_l[port q], Z = Y^-1
    ports = torch.arange(nl - E.np, nl)
    for f in s["freqs"]:
        w = 2 * math.pi * f
        M = E.product(torch.eye(nl, dtype=torch.complex128, device="cuda"), np.full(nl, w), "loop").T
        b = torch.zeros(nl, E.np, dtype=torch.complex128, device="cuda")
        b[ports, torch.arange(E.np)] = 1
        Z.append(torch.linalg.inv(torch.linalg.solve(M, b)[ports.cuda()]).cpu().numpy())
    return np.stack(Z)
