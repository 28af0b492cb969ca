"""The work a user of this framework has it do, as cases that can be timed one by one.

A user sets an operator up (a new mesh, or the next wavenumber of a sweep on a known mesh), applies
it and its preconditioners to blocks of vectors, solves for one or many excitations, takes the
bistatic RCS of the currents, and compresses the operator and applies the compressed form.  Every
case is one such call through the public Python API.  Meshes are the closed and open surfaces of
the tests and the benchmark (geodesic spheres, ellipsoids, tori, square plates; 480 to 30720
unknowns), jittered by the seed; right-hand-side blocks run from one column to the 64 of a serving
request.

Solves run to a residual of 1e-10, the setting used wherever currents are compared, so that a
current does not depend on where the last sweep of a loose solve happened to stop.  Operators that
are applied directly take the closed-form scaling alpha = sqrt(k), beta = 1/sqrt(k), gamma = k;
the estimated scaling (good to about 1e-3 by design) is timed in the setup and solve cases.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1803_08333_gb300 as rf

_CTX = []


def _context():
    if not _CTX:
        _CTX.append(rf.Context(0))
    return _CTX[0]


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # a small body probed once: launches and latency are all there is
        {"name": "apply_T_smallest", "kind": "apply", "which": "T", "mesh": "sphere", "n": 4, "ka": 1.0, "cols": 1},
        # the accurate RCS-grade application of the low-frequency benchmark's own mesh, one excitation
        {"name": "apply_A_one_largest", "kind": "apply", "which": "A", "mesh": "sphere", "n": 32, "ka": 0.1, "cols": 1},
        # a block of excitations through the accurate operator
        {"name": "apply_A_block", "kind": "apply", "which": "A", "mesh": "ellipsoid", "n": 16, "ka": 1.0, "cols": 16},
        # three excitations on an open plate of odd size: the preconditioner's middle operator
        {"name": "precondition_plate", "kind": "precondition", "which": "P_M", "mesh": "plate", "n": 51, "ka": 0.5,
         "cols": 3},
        # one plane wave on the level-3 sphere: the solve a single user waits for
        {"name": "solve_one", "kind": "solve", "mesh": "sphere", "n": 8, "ka": 1.0, "cols": 1},
        # one serving request of many plane waves on a mid-size body
        {"name": "solve_request", "kind": "solve", "mesh": "ellipsoid", "n": 18, "ka": 1.0, "cols": 24},
        # a body seen for the first time: topology, factors, matrices, estimated scaling
        {"name": "setup_new_mesh", "kind": "setup_mesh", "mesh": "sphere", "n": 20, "ka": 1.0},
        # the next wavenumber of a sweep on a known body
        {"name": "setup_wavenumber", "kind": "setup_k", "mesh": "sphere", "n": 24, "ka": 0.1},
        # bistatic RCS on the two 181-angle cuts of the benchmark
        {"name": "rcs_cuts", "kind": "rcs", "mesh": "sphere", "n": 32, "ka": 1.0, "cols": 1, "dirs": 362},
        # RCS of a whole block of excitations
        {"name": "rcs_block", "kind": "rcs", "mesh": "torus", "n": 40, "ka": 2.0, "cols": 23, "dirs": 91},
        # compression of a body's operator (then one product with each part, which is its result)
        {"name": "compress", "kind": "compress", "mesh": "sphere", "n": 16, "ka": 1e-3, "cols": 1},
        # products with the compressed operator of a larger body
        {"name": "compressed_products", "kind": "compressed", "mesh": "ellipsoid", "n": 24, "ka": 1e-3, "cols": 8},
    ]


_RANGE = {  # mesh sizes of each kind: (smallest, largest) frequency of a geodesic sphere
    "apply": (4, 32), "precondition": (4, 32), "solve": (4, 20), "setup_mesh": (6, 20), "setup_k": (6, 24),
    "rcs": (6, 32), "compress": (6, 16), "compressed": (6, 24),
}


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(sorted(_RANGE))
    lo, hi = _RANGE[kind]
    f = math.exp(rng.uniform(math.log(lo), math.log(hi)))  # spheres of frequency f have 20 f^2 cells
    mesh = rng.choice(["sphere", "ellipsoid", "torus", "plate"])
    if kind == "solve" and mesh == "plate":  # whole solves: closed bodies
        mesh = "torus"
    # tori of 2 n (n // 2) cells, plates of 2 n^2 cells: as many cells as the sphere, or fewer
    n = {"sphere": int(f), "ellipsoid": int(f), "torus": max(6, int(math.sqrt(20.0) * f)),
         "plate": max(5, int(math.sqrt(10.0) * f))}[mesh]
    case = {"kind": kind, "mesh": mesh, "n": n}
    case["ka"] = round(math.exp(rng.uniform(math.log(1e-3), math.log(1.5))), 6)
    cells = 20 * f * f
    if kind in ("apply", "precondition"):
        case["which"] = rng.choice(["T", "T_A", "T_ADJ", "T_PHI", "A"] if kind == "apply" else
                                   ["P_O", "P_M", "P_SIGMA", "P_LAMBDAH"])
        case["cols"] = log_int(1, 64 if cells <= 2000 else (16 if cells <= 6000 else 2))
    elif kind == "solve":
        case["ka"] = round(rng.uniform(0.1, 1.2), 4)
        case["cols"] = log_int(1, 64 if cells <= 2000 else 16)
    elif kind == "rcs":
        case["cols"] = log_int(1, 32 if cells <= 3200 else (8 if cells <= 8000 else 1))
        case["dirs"] = log_int(5, 362 if case["cols"] <= 2 else 91)
    elif kind in ("compress", "compressed"):
        case["ka"] = round(math.exp(rng.uniform(math.log(1e-5), math.log(1.0))), 7)
        case["cols"] = 1 if kind == "compress" else log_int(1, 8)
    return case


# ---------------------------------------------------------------- seeded surfaces
def _sphere(n, rng):
    t = (1.0 + 5.0**0.5) / 2.0
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    d = np.linalg.norm(v[:, None] - v[None], axis=-1)
    near = d < 1.2  # the five neighbours of a corner of the icosahedron
    faces = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
             if near[a, b] and near[b, c] and near[a, c]]
    ij = [(i, j) for i in range(n + 1) for j in range(n + 1 - i)]
    at = {p: q for q, p in enumerate(ij)}
    w = np.array([(n - i - j, i, j) for i, j in ij], dtype=np.float64) / n
    local = []
    for i in range(n):
        for j in range(n - i):
            local.append((at[i, j], at[i + 1, j], at[i, j + 1]))
            if i + j + 1 < n:
                local.append((at[i + 1, j], at[i + 1, j + 1], at[i, j + 1]))
    pts = np.concatenate([w @ v[list(f)] for f in faces])
    tris = np.concatenate([np.array(local) + q * len(ij) for q in range(len(faces))])
    _, first, back = np.unique(np.round(pts * 1e7).astype(np.int64), axis=0, return_index=True, return_inverse=True)
    pts, tris = pts[first], back.reshape(-1)[tris]
    pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    h = 1.1 / n  # about the mean edge
    pts = pts + 0.03 * h * rng.uniform(-0.6, 0.6, pts.shape)
    pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    a, b, c = pts[tris[:, 0]], pts[tris[:, 1]], pts[tris[:, 2]]
    flip = np.einsum("ij,ij->i", np.cross(b - a, c - a), a + b + c) < 0
    tris[flip] = tris[flip][:, [0, 2, 1]]
    return pts, tris


def _mesh(case, seed):
    rng = np.random.default_rng(seed)
    n = case["n"]
    if case["mesh"] in ("sphere", "ellipsoid"):
        v, t = _sphere(n, rng)
        if case["mesh"] == "ellipsoid":
            v = v * np.array([1.0, 0.8, 0.6])
    elif case["mesh"] == "torus":
        m = max(3, n // 2)
        h = 2.0 * math.pi / n
        u, w = np.meshgrid(h * np.arange(n), 2.0 * math.pi / m * np.arange(m), indexing="ij")
        u = u + 0.03 * h * rng.uniform(-1, 1, u.shape)
        w = w + 0.03 * h * rng.uniform(-1, 1, w.shape)
        v = np.stack([(1 + 0.4 * np.cos(w)) * np.cos(u), (1 + 0.4 * np.cos(w)) * np.sin(u), 0.4 * np.sin(w)], -1)
        v = v.reshape(-1, 3)
        i, j = (q.reshape(-1) for q in np.meshgrid(np.arange(n), np.arange(m), indexing="ij"))
        a, b, c, d = (p % n * m + q % m for p, q in ((i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1)))
        t = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)])
    else:
        x, y = np.meshgrid(np.arange(n + 1) / n - 0.5, np.arange(n + 1) / n - 0.5, indexing="ij")
        inner = np.zeros(x.shape)
        inner[1:-1, 1:-1] = 0.03 / n
        x, y = x + inner * rng.uniform(-1, 1, x.shape), y + inner * rng.uniform(-1, 1, x.shape)
        v = np.stack([x, y, np.zeros_like(x)], -1).reshape(-1, 3)
        i, j = (q.reshape(-1) for q in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
        a, b, c, d = (p * (n + 1) + q for p, q in ((i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1)))
        even = ((i + j) % 2 == 0)[:, None]
        t = np.concatenate([np.where(even, np.stack([a, b, c], 1), np.stack([a, b, d], 1)),
                            np.where(even, np.stack([a, c, d], 1), np.stack([b, c, d], 1))])
    return np.ascontiguousarray(v, dtype=np.float64), np.ascontiguousarray(t, dtype=np.int32)


def _waves(cols, seed):
    rng = np.random.default_rng([seed, 7])
    kh = rng.standard_normal((cols, 3))
    kh /= np.linalg.norm(kh, axis=1, keepdims=True)
    p = np.cross(kh, rng.standard_normal((cols, 3)))
    return kh, p / np.linalg.norm(p, axis=1, keepdims=True)


def _dirs(count, seed):
    """Unit directions of a few cuts: the polar angle runs over half a turn per cut."""
    rng = np.random.default_rng([seed, 8])
    th = np.pi * (np.arange(count) % 181) / 180.0
    ph = rng.uniform(0, np.pi) + 0.5 * np.pi * (np.arange(count) // 181)
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)


def _block(cols, n, seed, what=0):
    rng = np.random.default_rng([seed, 9, what])
    return rng.standard_normal((cols, n)) + 1j * rng.standard_normal((cols, n))


def _sizes(case):
    """(unknowns, cells, loops) of the case's mesh."""
    n = case["n"]
    if case["mesh"] in ("sphere", "ellipsoid"):
        return 30 * n * n, 20 * n * n, 10 * n * n + 2
    if case["mesh"] == "torus":
        c = 2 * n * max(3, n // 2)
        return 3 * c // 2, c, c // 2
    return 3 * n * n - 2 * n, 2 * n * n, (n - 1) ** 2


# ---------------------------------------------------------------- one pass
def prepare(case, seed):
    ctx = _context()
    kind, k = case["kind"], case["ka"]
    v, t = _mesh(case, seed)
    st = {"case": case, "ctx": ctx, "v": v, "t": t, "k": k}
    N, C, _ = _sizes(case)
    ctx.clear_cache()  # factors of bodies that no operator holds any more
    if kind == "setup_mesh":
        return st
    if kind == "setup_k":
        # the sweep's previous wavenumber: its operator is what the next one starts from
        st["before"] = rf.Operator(ctx, v, t, 10.0 * k)
        return st
    if kind == "solve":
        st["op"] = rf.Operator(ctx, v, t, k)
        st["e"] = st["op"].rhs_planewave(*_waves(case["cols"], seed))
        return st
    st["op"] = rf.Operator(ctx, v, t, k, scaling="k")
    if kind == "rcs":  # smooth surface currents, as a solve gives them
        st["x"] = st["op"].rhs_planewave(*_waves(case["cols"], seed))
        st["dirs"] = _dirs(case["dirs"], seed)
        return st
    st["x"] = torch.from_numpy(_block(case["cols"], N, seed)).cuda()
    if kind in ("compress", "compressed"):
        st["s"] = torch.from_numpy(_block(case["cols"], C, seed, 1)).cuda()
    if kind == "compressed":
        st["h"] = rf.Compressed(st["op"], eps=1e-4)
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "apply":
        return st["op"].apply(case["which"], st["x"])
    if kind == "precondition":
        return st["op"].precondition(case["which"], st["x"])
    if kind == "solve":
        return st["op"].solve(st["e"], tol=1e-10)[0]
    if kind == "rcs":
        return st["op"].farfield(st["x"], st["dirs"])
    if kind == "setup_mesh":
        st["ctx"].clear_cache()  # this body has not been seen before
        op = rf.Operator(st["ctx"], st["v"], st["t"], st["k"])
        out = {"T_A": op.export("T_A"), "V": op.export("V"), "lplus": op.export("LPLUS"),
               "gll_inv": op.export("GLL_INV"), "scaling": np.array(op.scaling, dtype=np.float32)}
        op.close()
        return out
    if kind == "setup_k":
        op = rf.Operator(st["ctx"], st["v"], st["t"], st["k"], scaling_start=st["before"])
        out = {"T_A": op.export("T_A"), "V": op.export("V"), "scaling": np.array(op.scaling, dtype=np.float32)}
        op.close()
        return out
    h = st["h"] if kind == "compressed" else rf.Compressed(st["op"], eps=1e-4)
    out = {"T_A": h.apply("T_A", st["x"]), "V": h.apply("V", st["s"])}
    if kind == "compress":
        h.close()
    return out


def work(case):
    """Bytes and operations of one pass.  A complex64 entry takes 8 bytes, a factor entry 8 (two FP32
    words), both matrices and factors are symmetric (half of them has to be read), a real
    multiply-add counts 2."""
    N, C, L = map(float, _sizes(case))
    kind, r = case["kind"], float(case.get("cols", 1))
    ta, v, lp, gl = 4 * N * N, 4 * C * C, 4 * C * C, 4 * L * L  # half of each
    fta, fv, flp, fgl = 8 * N * N, 8 * C * C, 4 * C * C, 4 * L * L  # per column
    if kind == "apply":
        b, f = {"T_A": (ta, fta), "T_PHI": (v, fv), "T": (ta + v, fta + fv), "T_ADJ": (ta + v, fta + fv),
                "A": (ta + v + lp + gl, 2 * fta + 2 * fv + 4 * flp + fgl)}[case["which"]]
        return {"bytes": b + 32 * N * r, "flops": f * r}
    if kind == "precondition":
        b, f = {"P_M": (lp + gl, 2 * flp + fgl)}.get(case["which"], (lp, flp))
        return {"bytes": b + 32 * N * r, "flops": f * r}
    if kind == "solve":  # some twenty applications to 1e-10, the operator read once
        return {"bytes": ta + v + lp + gl + 32 * N * r, "flops": 20 * r * (2 * fta + 2 * fv + 4 * flp + fgl)}
    if kind == "rcs":  # a phase per (direction, cell) and quadrature point, the current sums per column
        return {"bytes": 16 * N * r + 240 * C + 8 * r * case["dirs"], "flops": case["dirs"] * C * (150 + 48 * r)}
    pairs = C * C / 2  # 7 x 7 points, about 20 operations each
    if kind == "setup_k":
        return {"bytes": 8 * N * N + 8 * C * C, "flops": pairs * 49 * 20}
    if kind == "setup_mesh":  # the matrices, and one dense inverse of each factor by products
        return {"bytes": 8 * N * N + 8 * C * C + 8 * C * C + 8 * L * L, "flops": pairs * 49 * 20 + 2 * C**3 + 2 * L**3}
    # compressed: about 64 stored entries per n log2 n, halved by symmetry in both products
    e = sum(min(n * n / 2, 64 * n * math.log2(n)) for n in (N, C))
    if kind == "compress":
        return {"bytes": 8 * e + 32 * (N + C) * r, "flops": 30 * e}
    return {"bytes": 8 * e + 32 * (N + C) * r, "flops": 16 * e * r}


# ---------------------------------------------------------------- the same in 64 bits
_A1, _B1 = (6 - math.sqrt(15)) / 21, (6 + math.sqrt(15)) / 21
_WA, _WB = (155 - math.sqrt(15)) / 1200, (155 + math.sqrt(15)) / 1200
_BARY = [[1 / 3] * 3] + [[x if i != z else 1 - 2 * x for i in range(3)] for x in (_A1, _B1) for z in (2, 1, 0)]
_WTS = [9 / 40] + [_WA] * 3 + [_WB] * 3


class _Surface:
    """RWG functions of a triangulation in plain FP64: edges sorted by (lower, higher vertex), those of
    two cells only, + on the cell of lower index; loops on the vertices off the boundary."""

    def __init__(self, v, t):
        dev = "cuda"
        self.t = t.astype(np.int64)
        nc = len(t)
        loc = self.t[:, [[1, 2], [2, 0], [0, 1]]]  # the edge opposite each corner
        key = np.sort(loc, -1).reshape(-1, 2)
        uniq, inv, cnt = np.unique(key, axis=0, return_inverse=True, return_counts=True)
        inv = inv.reshape(-1)
        two = cnt == 2
        num = np.where(two, np.cumsum(two) - 1, -1)
        self.edge = num[inv].reshape(nc, 3)
        first = np.full(len(uniq), nc * 3, dtype=np.int64)
        np.minimum.at(first, inv, np.arange(3 * nc))
        self.sign = np.where(first[inv] == np.arange(3 * nc), 1.0, -1.0).reshape(nc, 3)
        self.N, self.nc, self.nv = int(two.sum()), nc, len(v)
        rim = np.zeros(len(v), bool)
        rim[uniq[~two].reshape(-1)] = True
        self.loops = np.cumsum(~rim) - 1
        self.loops[rim] = -1
        self.L = int((~rim).sum())
        # Lambda: +1 at the first, -1 at the second end of the edge as the + cell runs through it
        f = first[two]
        self.ends = loc.reshape(-1, 2)[f]
        self.X = torch.from_numpy(v).to(dev)
        self.P = self.X[torch.from_numpy(self.t).to(dev)]  # (nc, 3, 3)
        cr = torch.linalg.cross(self.P[:, 1] - self.P[:, 0], self.P[:, 2] - self.P[:, 0])
        self.area = 0.5 * cr.norm(dim=1)
        self.nrm = cr / cr.norm(dim=1, keepdim=True)
        self.cen = self.P.mean(1)
        self.bary = torch.tensor(_BARY, dtype=torch.float64, device=dev)
        self.w = torch.tensor(_WTS, dtype=torch.float64, device=dev)
        self.q = torch.einsum("qi,cia->cqa", self.bary, self.P)
        self.rho = self.q - self.cen[:, None]
        self.corner = self.P - self.cen[:, None]
        self.e = torch.from_numpy(self.edge).to(dev)
        self.s = torch.from_numpy(self.sign).to(dev)

    def sigma(self):
        S = torch.zeros((self.N + 1, self.nc), dtype=torch.float64, device="cuda")
        for i in range(3):
            at = torch.where(self.e[:, i] < 0, self.N, self.e[:, i])
            S[at, torch.arange(self.nc, device="cuda")] += self.s[:, i]
        return S[: self.N]

    def lam(self):
        M = torch.zeros((self.N, self.L + 1), dtype=torch.float64, device="cuda")
        for z, sg in ((0, 1.0), (1, -1.0)):
            c = self.loops[self.ends[:, z]]
            M[torch.arange(self.N, device="cuda"), torch.from_numpy(np.where(c < 0, self.L, c)).cuda()] += sg
        return M[:, : self.L]

    def mass(self):
        M = torch.zeros((self.L + 1) ** 2, dtype=torch.float64, device="cuda")
        l = torch.from_numpy(np.where(self.loops < 0, self.L, self.loops)[self.t]).cuda()
        for i in range(3):
            for j in range(3):
                M.index_add_(0, l[:, i] * (self.L + 1) + l[:, j], self.area / (6.0 if i == j else 12.0))
        return M.view(self.L + 1, self.L + 1)[: self.L, : self.L]

    def near_pairs(self):
        order = np.argsort(self.t.reshape(-1), kind="stable")
        vert, cell = self.t.reshape(-1)[order], order // 3
        start = np.searchsorted(vert, np.arange(self.nv + 1))
        got, most = [], int(np.diff(start).max())
        for a in range(most):
            for b in range(most):
                ok = (start[:-1] + max(a, b)) < start[1:]
                got.append(np.stack([cell[start[:-1][ok] + a], cell[start[:-1][ok] + b]], 1))
        p = np.concatenate(got)
        return torch.from_numpy(np.unique(p[p[:, 0] <= p[:, 1]], axis=0)).cuda()

    def _static(self, r, P, nrm):
        """int 1/R and int (r' - p)/R over the triangles P (m, 3, 3) from the points r (m, 7, 3), and the
        points p under r in the triangles' planes."""
        d = ((r - P[:, None, 0]) * nrm[:, None]).sum(-1)
        p = r - d[..., None] * nrm[:, None]
        S, V, ad = 0.0, 0.0, d.abs()
        for i in range(3):
            A, B = P[:, i], P[:, (i + 1) % 3]
            l = (B - A) / (B - A).norm(dim=1, keepdim=True)
            u = torch.linalg.cross(l, nrm)[:, None]
            l = l[:, None]
            lp, lm = ((B[:, None] - p) * l).sum(-1), ((A[:, None] - p) * l).sum(-1)
            p0 = ((A[:, None] - p) * u).sum(-1)
            r0 = p0 * p0 + d * d
            rp, rm = (lp * lp + r0).sqrt(), (lm * lm + r0).sqrt()
            up = torch.where(lp > 0, rp + lp, r0 / (rp - lp).clamp_min(1e-300))
            um = torch.where(lm > 0, rm + lm, r0 / (rm - lm).clamp_min(1e-300))
            scale = (B - A).square().sum(-1)[:, None]
            F = torch.where(r0 > 1e-30 * scale, (up / um.clamp_min(1e-300)).clamp_min(1e-300).log(), 0.0)
            at = torch.atan2(p0 * lp, r0 + ad * rp) - torch.atan2(p0 * lm, r0 + ad * rm)
            S = S + p0 * F - ad * torch.where(ad > 0, at, 0.0)
            V = V + (0.5 * (r0 * F + lp * rp - lm * rm))[..., None] * u
        return S, V, p

    def _near(self, o, i, k):
        """4 x 4 moments of (1, rho) x (1, rho') over outer cells o and inner cells i."""
        r = self.q[o]
        S, V, p = self._static(r, self.P[i], self.nrm[i])
        J = torch.cat([S[..., None], V + (p - self.cen[i][:, None]) * S[..., None]], -1) / (4 * math.pi) + 0j
        for j in range(7):
            R = (r - self.q[i, j][:, None]).norm(dim=-1)
            z = R < 1e-14
            Rs = torch.where(z, 1.0, R)
            h = torch.sin(0.5 * k * Rs)
            g = torch.complex(torch.where(z, 0.0, -2 * h * h / Rs), torch.where(z, k, torch.sin(k * Rs) / Rs))
            one = torch.cat([torch.ones_like(self.rho[i, j, :1]), self.rho[i, j]], -1)
            J = J + (self.w[j] * self.area[i] / (4 * math.pi))[:, None, None] * g[..., None] * one[:, None]
        W = torch.cat([torch.ones_like(self.rho[o][..., :1]), self.rho[o]], -1) * self.w[:, None]
        return torch.einsum("mqa,mqb->mab", W + 0j, J) * self.area[o][:, None, None]

    def assemble(self, k):
        """T_A and V, complex128."""
        nc, N = self.nc, self.N
        W = torch.cat([torch.ones_like(self.rho[..., :1]), self.rho], -1) * self.w[:, None] * self.area[:, None, None]
        pairs = self.near_pairs()
        s, t = pairs[:, 0], pairs[:, 1]
        M = 0.5 * (self._near(s, t, k) + self._near(t, s, k).transpose(1, 2))
        off = s != t
        ns, nt = torch.cat([s, t[off]]), torch.cat([t, s[off]])
        M = torch.cat([M, M[off].transpose(1, 2)])
        order = torch.argsort(ns)
        ns, nt, M = ns[order], nt[order], M[order]
        V = torch.empty((nc, nc), dtype=torch.complex128, device="cuda")
        TA = torch.zeros((N + 1, N + 1), dtype=torch.complex128, device="cuda")
        step = max(1, int(2.5e7) // (49 * nc))
        Wc = W + 0j
        e = torch.where(self.e < 0, N, self.e)
        for b in range(0, nc, step):
            z = min(nc, b + step)
            m = z - b
            R = torch.zeros((m * 7, nc * 7), dtype=torch.float64, device="cuda")
            for a in range(3):
                R += (self.q[b:z, :, a].reshape(-1, 1) - self.q[:, :, a].reshape(1, -1)).square()
            R = R.sqrt_().clamp_min_(1e-300)
            G = torch.polar(1.0 / (4 * math.pi * R), k * R)
            del R
            K = torch.einsum("xtp,tpb->xtb", G.view(m * 7, nc, 7), Wc).view(m, 7, nc, 4)
            K = torch.einsum("sqtb,sqa->stab", K, Wc[b:z])
            lo, hi = torch.searchsorted(ns, torch.tensor([b, z], device="cuda")).tolist()
            K[ns[lo:hi] - b, nt[lo:hi]] = M[lo:hi]
            K = K / (self.area[b:z, None, None, None] * self.area[None, :, None, None])
            V[b:z] = K[..., 0, 0]
            dot = K[..., 1, 1] + K[..., 2, 2] + K[..., 3, 3]
            for j in range(3):
                rows = torch.zeros((N + 1, nc), dtype=torch.complex128, device="cuda") if z == nc and b == 0 else None
                pj = self.corner[:, j] + 0j
                for i in range(3):
                    pi = self.corner[b:z, i] + 0j
                    c = dot - torch.einsum("sta,ta->st", K[..., 1:, 0], pj) - torch.einsum("stb,sb->st", K[..., 0, 1:], pi)
                    c = c + (pi @ pj.T) * K[..., 0, 0]
                    c = 0.25 * self.s[b:z, i, None] * self.s[None, :, j] * c
                    if rows is not None:
                        rows.index_add_(0, e[b:z, i], c)
                    else:
                        part = torch.zeros((m, N + 1), dtype=torch.complex128, device="cuda")
                        part.index_add_(1, e[:, j], c)
                        TA.index_add_(0, e[b:z, i], part)
                if rows is not None:
                    TA.index_add_(1, e[:, j], rows)
        return TA[:N, :N], V

    def plane_waves(self, k, kh, pol):
        kh, pol = torch.from_numpy(kh).cuda(), torch.from_numpy(pol).cuda()
        out = torch.zeros((len(kh), self.N + 1), dtype=torch.complex128, device="cuda")
        ph = torch.polar(torch.ones((), dtype=torch.float64, device="cuda").expand(len(kh), self.nc, 7),
                         k * torch.einsum("ra,cqa->rcq", kh, self.q))
        for i in range(3):
            f = torch.einsum("cqa,ra->rcq", self.q - self.P[:, i, None], pol) * self.w
            out.index_add_(1, torch.where(self.e[:, i] < 0, self.N, self.e[:, i]), 0.5 * self.s[:, i] * (f * ph).sum(-1))
        return out[:, : self.N]


def _application(sf, case, x):
    """The dense operators of the paper in 64 bits, applied to the columns of x (n x cols)."""
    k, which = case["ka"], case["which"]
    S = sf.sigma()
    if case["kind"] == "apply":
        TA, V = sf.assemble(k)
    mul = lambda M, z: torch.complex(M @ z.real, M @ z.imag)  # noqa: E731
    star, up = (lambda u: mul(S.T, u)), (lambda z: mul(S, z))  # noqa: E731

    def t_op(u, adj=False):
        a, v = (TA.conj(), V.conj()) if adj else (TA, V)
        s = -1.0 if adj else 1.0
        return 1j * k * s * (a @ u) + up(v @ star(u)) / (1j * k * s)

    if which == "T_A":
        return TA @ x
    if which == "T_PHI":
        return up(V @ star(x))
    if which in ("T", "T_ADJ"):
        return t_op(x, which == "T_ADJ")
    al, be, ga = math.sqrt(k), 1 / math.sqrt(k), k
    Lp = torch.linalg.inv(S.T @ S + 1.0 / sf.nc) - 1.0 / sf.nc
    p_s = lambda u: up(mul(Lp, star(u)))  # noqa: E731

    def p_o(u, sg=1.0):
        y = p_s(u)
        return (u - y) / al + sg * 1j * y / be

    def p_m(u):
        Lam, G = sf.lam(), sf.mass()
        z = mul(Lp, star(u))
        y = mul(Lam, mul(torch.linalg.inv(G), mul(Lam.T, u))) / al**2
        return y + (u - up(z)) / ga + up(mul(Lp, sf.area[:, None] * z)) / be**2

    if which == "P_SIGMA":
        return p_s(x)
    if which == "P_LAMBDAH":
        return x - p_s(x)
    if which == "P_O":
        return p_o(x)
    if which == "P_M":
        return p_m(x)
    return p_o(t_op(p_m(t_op(p_o(x))), True), -1.0)


def exact(case, seed):
    N, C, _ = _sizes(case)
    kind, k = case["kind"], case["ka"]
    if N > 18000 and kind != "rcs":
        return None  # dense 64-bit matrices of this size take too long
    sf = _Surface(*_mesh(case, seed))
    if kind in ("apply", "precondition"):
        if case["which"] == "A" and k < 0.05:
            return None  # the dense form cancels at low frequency
        x = torch.from_numpy(_block(case["cols"], N, seed)).cuda()
        return _application(sf, case, x.T).T.contiguous()
    if kind == "solve":
        if N > 8000:
            return None
        TA, V = sf.assemble(k)
        S = sf.sigma() + 0j
        T = 1j * k * TA + S @ V @ S.T / (1j * k)
        e = sf.plane_waves(k, *_waves(case["cols"], seed))
        return torch.linalg.solve(T, -e.T).T.contiguous()
    if kind == "rcs":
        x = sf.plane_waves(k, *_waves(case["cols"], seed))
        x = torch.cat([x, torch.zeros_like(x[:, :1])], 1)
        u = torch.from_numpy(_dirs(case["dirs"], seed)).cuda()
        J = 0.0
        for i in range(3):
            c = 0.5 * sf.s[:, i] * x[:, torch.where(sf.e[:, i] < 0, N, sf.e[:, i])]
            J = J + c[:, :, None, None] * ((sf.q - sf.P[:, i, None]) * sf.w[:, None])[None]
        J = J.reshape(x.shape[0], -1, 3).permute(1, 0, 2).reshape(-1, 3 * x.shape[0])
        F = []
        for b in range(0, len(u), 16):
            a = -k * (u[b : b + 16] @ sf.q.reshape(-1, 3).T)
            F.append(torch.polar(torch.ones_like(a), a) @ J)
        F = torch.cat(F).view(len(u), x.shape[0], 3).transpose(0, 1)
        F = F - (F * u).sum(-1, keepdim=True) * u
        return (10.0 * torch.log10(k * k / (4 * math.pi) * F.abs().square().sum(-1))).cpu().numpy()
    TA, V = sf.assemble(k)
    if kind in ("compress", "compressed"):
        x = torch.from_numpy(_block(case["cols"], N, seed)).cuda()
        s = torch.from_numpy(_block(case["cols"], C, seed, 1)).cuda()
        return {"T_A": (TA @ x.T).T.contiguous(), "V": (V @ s.T).T.contiguous()}
    out = {"T_A": TA, "V": V, "scaling": None}
    if kind == "setup_mesh":
        S = sf.sigma()
        out["lplus"] = torch.linalg.inv(S.T @ S + 1.0 / sf.nc) - 1.0 / sf.nc
        out["gll_inv"] = torch.linalg.inv(sf.mass())
    return out
