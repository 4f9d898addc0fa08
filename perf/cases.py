"""What is timed: calls of the library's entry points at the sizes its users have.

A user meshes a perfectly conducting body at lambda / 9, sets up a context
(grid spacing lambda / 10, 27-point stencils, near radius three spacings) and
then calls products, solves and far fields on it, many times.  Setup belongs
to ``prepare``; ``run`` is one call.  Bodies are the square plates and the
spheres of the repository's configurations (0.5 to 32 wavelengths) and
rectangular plates; spheres are closed and may use the combined-field
equation.  Sizes between the round ones are as common as the round ones (a
frequency sweep changes every length), so several listed cases have padded
grid lengths that are no power-of-two multiple of 45 or 81.

``exact`` is the method in 64 bits, in plain torch and numpy: RWG functions,
moment-matching weights, Green's function on the zero-padded grid, near
entries with the singularity taken out, and the four steps of the product.
"""

import functools
import math

import numpy as np
import torch

import paper_1010_1456_gb300 as g

K = 2.0 * math.pi  # lengths are in wavelengths
H = 0.1            # grid spacing
M = 2              # stencil order: 27 nodes
EDGE = 9.0         # mesh edges per wavelength
ALPHA = 0.6        # weight of the electric-field equation in the combined one
ETA0 = 376.730313668
PREC = {"c64": g.AIM_C64, "c128": g.AIM_C128, "f64": g.AIM_C128_F64}


def listed():
    return [
        # the smallest configuration: one product of a 1 lambda plate, FP64-accurate (latency, launches)
        {"name": "plate1_c128", "op": "product", "body": "plate", "size": 1.0, "cfie": False, "prec": "c128", "nrhs": 1},
        # a request of the serving stream: an open plate with a few incidence angles, the solver's inner product
        {"name": "plate5_c64_x4", "op": "product", "body": "plate", "size": 5.0, "cfie": False, "prec": "c64", "nrhs": 4},
        # a small closed body with the combined-field equation, as the serving stream solves it
        {"name": "sphere1.5_cfie_c64_x8", "op": "product", "body": "sphere", "size": 1.5, "cfie": True, "prec": "c64", "nrhs": 8},
        # many small requests at once: eight plates of 0.8 to 1.2 lambda in one pack
        {"name": "pack8_c64", "op": "pack", "body": "plate", "size": 0.8, "step": 0.05, "count": 8, "cfie": False, "nrhs": 2},
        # the plain single-right-hand-side configuration: sphere of 4 lambda, FP64-accurate
        {"name": "sphere4_c128", "op": "product", "body": "sphere", "size": 4.0, "cfie": False, "prec": "c128", "nrhs": 1},
        # the native FP64 path
        {"name": "sphere2_f64", "op": "product", "body": "sphere", "size": 2.0, "cfie": False, "prec": "f64", "nrhs": 1},
        # the batched mixed-precision configuration: 32 lambda plate, 64 incidences
        {"name": "plate32_c64_x64", "op": "product", "body": "plate", "size": 32.0, "cfie": False, "prec": "c64", "nrhs": 64},
        # an ordinary closed body between the round sizes, combined-field equation
        {"name": "sphere7_cfie_c64_x4", "op": "product", "body": "sphere", "size": 7.0, "cfie": True, "prec": "c64", "nrhs": 4},
        # the large configuration: sphere of 16 lambda, four directions in two polarisations
        {"name": "sphere16_c64_x8", "op": "product", "body": "sphere", "size": 16.0, "cfie": False, "prec": "c64", "nrhs": 8},
        # a call with host vectors, copies included (ragged number of right-hand sides)
        {"name": "plate12_c64_x17_host", "op": "host", "body": "plate", "size": 12.0, "cfie": False, "prec": "c64", "nrhs": 17},
        # a whole solve: combined-field sphere, two polarisations, FP64-accurate products (the default precision)
        {"name": "sphere2_cfie_solve", "op": "solve", "body": "sphere", "size": 2.0, "cfie": True, "prec": "c128", "nrhs": 2},
        # the bistatic pattern of two polarisations on the error measure's direction grid
        {"name": "sphere2_rcs_x2", "op": "rcs", "body": "sphere", "size": 2.0, "cfie": False, "nrhs": 2, "n_theta": 64},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    what = rng.random()
    if what < 0.68:
        body = rng.choice(["plate", "sphere", "strip"])
        prec = rng.choice(["c64", "c64", "c64", "c128", "f64"])
        # right-hand sides, then the largest body whose padded grids stay under 6 GB
        nrhs = int(round(_log(rng, 1, 64 if prec == "c64" else 8)))
        room = 6e9 / (4 * nrhs * (8 if prec == "c64" else 16))
        if body == "sphere":
            top = min(12.0, ((room / 2.0) ** (1.0 / 3.0) - 4) / 32.0)
            case = {"size": round(_log(rng, 0.5, max(0.6, top)), 2), "cfie": rng.random() < 0.5}
        else:
            top = min(32.0, (math.sqrt(room) - 6) / 20.0)
            case = {"size": round(_log(rng, 0.7, max(0.8, top)), 2), "cfie": False}
        if body == "strip":
            case["other"] = round(max(0.5, case["size"] * _log(rng, 0.1, 0.9)), 2)
        return {"op": "host" if rng.random() < 0.15 else "product", "body": body, "prec": prec, "nrhs": nrhs, **case}
    if what < 0.8:
        body = rng.choice(["plate", "sphere"])
        return {"op": "pack", "body": body, "size": round(rng.uniform(0.4, 0.8), 3), "step": round(rng.uniform(0.02, 0.09), 3),
                "count": rng.randint(2, 10), "cfie": body == "sphere", "nrhs": rng.randint(1, 4)}
    if what < 0.9:
        return {"op": "solve", "body": "sphere", "size": round(_log(rng, 0.5, 3.0), 2), "cfie": True, "prec": "c128",
                "nrhs": rng.randint(1, 4)}
    return {"op": "rcs", "body": rng.choice(["plate", "sphere"]), "size": round(_log(rng, 0.7, 3.0), 2), "cfie": False,
            "nrhs": rng.randint(1, 3), "n_theta": rng.randint(20, 90)}


# ---------------------------------------------------------------- meshes
def _rect(sx, sy):
    nx, ny = max(2, round(EDGE * sx)), max(2, round(EDGE * sy))
    tx = np.arange(nx + 1) * (sx / nx) - 0.5 * sx
    ty = np.arange(ny + 1) * (sy / ny) - 0.5 * sy
    X, Y = np.meshgrid(tx, ty, indexing="xy")
    verts = np.stack([X.ravel(), Y.ravel(), np.zeros(X.size)], axis=1)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny), indexing="xy"))
    v00 = j * (nx + 1) + i
    v01 = v00 + nx + 1
    tris = np.empty((2 * nx * ny, 3), dtype=np.int32)
    tris[0::2] = np.stack([v00, v00 + 1, v01 + 1], axis=1)
    tris[1::2] = np.stack([v00, v01 + 1, v01], axis=1)
    return verts, tris


def _sphere(radius):
    """Icosahedron with every face cut into f^2 triangles, pushed out to the sphere; outward order."""
    f = max(1, math.ceil(1.1755 * radius * EDGE - 1e-9))
    p = (1.0 + math.sqrt(5.0)) / 2.0
    iv = np.array([(0, a, b * p) for a in (-1, 1) for b in (-1, 1)] + [(a, b * p, 0) for a in (-1, 1) for b in (-1, 1)]
                  + [(b * p, 0, a) for a in (-1, 1) for b in (-1, 1)], dtype=np.float64)
    near = np.abs(((iv[:, None] - iv[None]) ** 2).sum(-1) - 4.0) < 1e-9
    faces = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
             if near[a, b] and near[b, c] and near[a, c]]
    faces = [(a, b, c) if np.dot(np.cross(iv[b] - iv[a], iv[c] - iv[a]), iv[a]) > 0 else (a, c, b) for a, b, c in faces]
    ij = np.array([(i, j) for i in range(f + 1) for j in range(f + 1 - i)])
    at = -np.ones((f + 2, f + 2), dtype=np.int64)
    at[ij[:, 0], ij[:, 1]] = np.arange(len(ij))
    low = ij[ij.sum(1) < f]
    up = ij[ij.sum(1) < f - 1]
    small = np.concatenate([
        np.stack([at[low[:, 0], low[:, 1]], at[low[:, 0] + 1, low[:, 1]], at[low[:, 0], low[:, 1] + 1]], axis=1),
        np.stack([at[up[:, 0] + 1, up[:, 1]], at[up[:, 0] + 1, up[:, 1] + 1], at[up[:, 0], up[:, 1] + 1]], axis=1)])
    # integer weights of the three corners identify a point shared by faces
    keys, tris = [], []
    for n, (a, b, c) in enumerate(faces):
        w = np.zeros((len(ij), 12), dtype=np.int16)
        w[:, a], w[:, b], w[:, c] = f - ij.sum(1), ij[:, 0], ij[:, 1]
        keys.append(w)
        tris.append(small + n * len(ij))
    keys = np.concatenate(keys)
    corner = keys.astype(np.int64)
    code = np.zeros(len(keys), dtype=np.int64)  # at most three corners: their numbers and two weights
    order = np.argsort(~(corner > 0), axis=1, kind="stable")[:, :3]
    for q in range(3):
        code = (code * 13 + order[:, q] * (np.take_along_axis(corner, order[:, q:q + 1], 1)[:, 0] > 0)) * (f + 1)
        code += np.take_along_axis(corner, order[:, q:q + 1], 1)[:, 0]
    _, first, back = np.unique(code, return_index=True, return_inverse=True)
    pts = (keys[first].astype(np.float64) / f) @ iv
    pts *= radius / np.sqrt((pts * pts).sum(1))[:, None]
    return pts, back.ravel()[np.concatenate(tris)].astype(np.int32)


@functools.lru_cache(maxsize=4)
def _mesh(body, size, other=None):
    if body == "sphere":
        return _sphere(size)
    return _rect(size, size if body == "plate" else other)


def _meshes(case):
    if case["op"] == "pack":
        return [_mesh(case["body"], case["size"] + i * case["step"]) for i in range(case["count"])]
    return [_mesh(case["body"], case["size"], case.get("other"))]


# ---------------------------------------------------------------- inputs
def _vector(n, N, seed, dtype):
    """Currents of a Krylov iteration: no structure along the numbering, unit variance."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn((n, N), generator=gen, dtype=torch.complex128, device="cuda").to(dtype)


def _waves(n, seed):
    """Plane waves from n random directions, each with a random polarisation across it."""
    rng = np.random.default_rng(seed)
    k = rng.standard_normal((n, 3))
    k /= np.linalg.norm(k, axis=1, keepdims=True)
    p = np.cross(k, rng.standard_normal((n, 3)))
    return k, p / np.linalg.norm(p, axis=1, keepdims=True)


def _directions(case):
    """Gauss nodes in cos(theta) and uniform ones in phi, as the error measure takes them."""
    mu, _ = np.polynomial.legendre.leggauss(case["n_theta"])
    phi = (np.arange(2 * case["n_theta"]) + 0.5) * (math.pi / case["n_theta"])
    T, P = np.meshgrid(np.arccos(mu), phi, indexing="ij")
    return T.ravel(), P.ravel()


def _dtype(case):
    return torch.complex64 if case.get("prec", "c64") == "c64" else torch.complex128


def prepare(case, seed):
    ctxs = [g.aim_setup(v, t, K, H, M=M, max_rhs=case["nrhs"], cfie_alpha=ALPHA if case["cfie"] else 1.0,
                        precision=PREC[case.get("prec", "c64")]) for v, t in _meshes(case)]
    state = {"case": case, "ctx": ctxs[0]}
    N, n = ctxs[0].N, case["nrhs"]
    if case["op"] == "pack":
        state["pack"] = g.aim_pack_create(ctxs, [n] * len(ctxs))
        state["x"] = state["pack"].pack([_vector(n, c.N, seed * 16 + i, torch.complex64) for i, c in enumerate(ctxs)])
    elif case["op"] == "solve":
        k, p = _waves(n, seed)
        state["V"] = g.aim_rhs_planewave(ctxs[0], k, p)
    elif case["op"] == "host":
        state["x"] = _vector(n, N, seed, _dtype(case)).cpu().pin_memory()
        state["y"] = torch.empty_like(state["x"]).pin_memory()
    else:
        state["x"] = _vector(n, N, seed, torch.complex128 if case["op"] == "rcs" else _dtype(case))
    if case["op"] == "rcs":
        state["angles"] = _directions(case)
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["op"] == "product":
        return g.aim_matvec(ctx, state["x"], precision=PREC[case["prec"]])
    if case["op"] == "host":
        return g.aim_matvec_host(ctx, state["x"], precision=PREC[case["prec"]], out=state["y"])
    if case["op"] == "pack":
        return g.aim_pack_matvec(state["pack"], state["x"])
    if case["op"] == "solve":
        return g.aim_solve(ctx, state["V"], tol=1e-6)[0]
    return list(g.aim_rcs(ctx, state["x"], *state["angles"]))


# ---------------------------------------------------------------- work
def _smooth(m):
    while True:
        x = m
        for p in (2, 3, 5):
            while x % p == 0:
                x //= p
        if x == 1:
            return m
        m += 1


def _unknowns(tris):
    e = np.sort(np.concatenate([tris[:, [0, 1]], tris[:, [1, 2]], tris[:, [2, 0]]]).astype(np.int64), axis=1)
    _, count = np.unique(e[:, 0] * (1 << 32) + e[:, 1], return_counts=True)
    return int((count == 2).sum())


def _product_work(verts, tris, case):
    """One product: vectors, near entries, weights and spectrum once; the pruned transforms, the sparse parts."""
    B, e = case["nrhs"], 8 if _dtype(case) == torch.complex64 else 16
    N = _unknowns(tris)
    planar = case["body"] != "sphere"
    S = 9 if planar else 27
    n = np.floor((verts.max(0) - verts.min(0)) / H).astype(int) + M + 1
    n[2] = 1 if planar else n[2]
    L = np.array([_smooth(max(1, 2 * int(v) - 1)) for v in n])
    # unknowns within the near radius of one: three edges per two triangles of area sqrt(3)/4 (plate: 1/2) edge^2
    per = 3.0 * EDGE ** 2 if planar else 1.5 * EDGE ** 2 / (math.sqrt(3) / 4)
    nnz = N * min(N, math.pi * (3 * H) ** 2 * per)
    comps = 7 if case["cfie"] else 4
    lg = [5.0 * v * math.log2(v) if v > 1 else 0.0 for v in L]
    fft = 4 * B * 2 * (n[0] * n[1] * lg[2] + n[0] * L[2] * lg[1] + L[1] * L[2] * lg[0]) + 4 * B * 6.0 * L.prod()
    return (2.0 * B * N * e + nnz * (e + 4) + N * S * comps * e / 2 + np.prod(L // 2 + 1) * e,
            fft + B * (N * S * 4.0 * (4 + comps) + 8.0 * nnz))


def work(case):
    if case["op"] == "rcs":
        verts, tris = _meshes(case)[0]
        points, dirs = 9.0 * len(tris), 2.0 * case["n_theta"] ** 2
        # a phase (a dot product, a sine and a cosine: about 40 operations) for every pair, then 12 products a right-hand side
        return {"bytes": 16.0 * case["nrhs"] * _unknowns(tris) + dirs * 16 * (1 + case["nrhs"]) + 24.0 * len(verts),
                "flops": points * dirs * (40.0 + 24.0 * case["nrhs"])}
    each = [_product_work(v, t, case) for v, t in _meshes(case)]
    # a solve to 1e-6 of a combined-field sphere of this range takes some 50 products
    times = 50.0 if case["op"] == "solve" else 1.0
    return {"bytes": times * float(sum(b for b, _ in each)), "flops": times * float(sum(f for _, f in each))}


# ---------------------------------------------------------------- the method in 64 bits
DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64, C128 = torch.float64, torch.complex128


def _rule(n):
    """Collapsed Gauss rule on a triangle: barycentric coordinates [q, 3] and weights that sum to one."""
    s, w = np.polynomial.legendre.leggauss(n)
    s, w = 0.5 * (s + 1.0), 0.5 * w
    S, T = (a.ravel() for a in np.meshgrid(s, s, indexing="ij"))
    W = (2.0 * w[:, None] * w[None, :]).ravel() * (1.0 - S)
    x2 = T * (1.0 - S)
    return torch.tensor(np.stack([1.0 - S - x2, S, x2], axis=1), device=DEV), torch.tensor(W, device=DEV)


class _Exact:
    """The AIM operator of one body in 64 bits."""

    def __init__(self, verts, tris, alpha):
        self.alpha = alpha
        tris = tris.astype(np.int64)
        ends = np.concatenate([tris[:, [1, 2]], tris[:, [2, 0]], tris[:, [0, 1]]])  # the edge across from slot 0, 1, 2
        ends.sort(axis=1)
        tri, slot = np.tile(np.arange(len(tris)), 3), np.repeat(np.arange(3), len(tris))
        order = np.lexsort((tri, ends[:, 1], ends[:, 0]))
        e, tri, slot = ends[order], tri[order], slot[order]
        two = np.nonzero((e[1:] == e[:-1]).all(1))[0]
        d = verts[e[two, 1]] - verts[e[two, 0]]
        self.N = len(two)
        to = lambda a: torch.tensor(a, device=DEV)  # noqa: E731
        self.tv = to(verts)[to(tris)]  # [T, 3, 3]
        self.tris = to(tris)
        self.length = to(np.sqrt((d * d).sum(1)))
        centre = (verts[e[two, 0]] + verts[e[two, 1]]) * 0.5
        self.centre = to(centre)
        self.half = [(to(tri[two]), to(slot[two]), 1.0), (to(tri[two + 1]), to(slot[two + 1]), -1.0)]
        nrm = torch.linalg.cross(self.tv[:, 1] - self.tv[:, 0], self.tv[:, 2] - self.tv[:, 0])
        size = nrm.square().sum(-1).sqrt()
        self.area, self.normal = 0.5 * size, nrm / size[:, None]
        anc = to(np.floor(centre / H - 0.5 * (M - 1)).astype(np.int64))  # a true division, on the host
        lo = anc.amin(0)
        self.n = (anc.amax(0) + M - lo + 1).tolist()
        self.anc = anc
        r = torch.arange(M + 1, device=DEV)
        kk, jj, ii = torch.meshgrid(r, r, r, indexing="ij")
        self.off = torch.stack([ii.ravel(), jj.ravel(), kk.ravel()], 1)
        node = (anc - lo)[:, None, :] + self.off
        self.node = (node[..., 2] * self.n[1] + node[..., 1]) * self.n[0] + node[..., 0]
        self._weights()
        self._near()
        self._spectrum()

    def _halves(self, n):
        """Per half: points [N, q, 3], the function's values there and the weights of the rule times the area."""
        bary, w = _rule(n)
        for tri, slot, sign in self.half:
            tv, area = self.tv[tri], self.area[tri]
            pts = torch.einsum("qv,nvx->nqx", bary, tv)
            free = tv[torch.arange(self.N, device=DEV), slot]
            f = (sign * self.length / (2.0 * area))[:, None, None] * (pts - free[:, None, :])
            yield tri, sign, area, pts, f, area[:, None] * w

    def _weights(self):
        """Moment-matching weights in Lagrange form: the integral of each function against the nodes' polynomials."""
        P = M + 1
        lam = torch.zeros((self.N, 4, P ** 3), dtype=F64, device=DEV)
        mf = torch.zeros((self.N, 3, P ** 3), dtype=F64, device=DEV)
        for tri, sign, area, pts, f, wa in self._halves((3 * M + 4) // 2):
            s = pts / H - self.anc[:, None, :]
            l, d = [], []
            for i in range(P):
                val, der = torch.ones_like(s), torch.zeros_like(s)
                for j in range(P):
                    if j != i:
                        der = (der * (s - j) + val) / (i - j)
                        val = val * (s - j) / (i - j)
                l.append(val)
                d.append(der / H)
            div = (sign * self.length / area)[:, None]
            for u in range(P ** 3):
                i, j, k = (int(v) for v in self.off[u])
                x, y, z = l[i][..., 0], l[j][..., 1], l[k][..., 2]
                b = wa * x * y * z
                lam[:, :3, u] += (b[..., None] * f).sum(1)
                lam[:, 3, u] += (b * div).sum(1)
                if self.alpha != 1.0:
                    grad = torch.stack([d[i][..., 0] * y * z, x * d[j][..., 1] * z, x * y * d[k][..., 2]], -1)
                    nrm = self.normal[tri]
                    fg, ng = (f * grad).sum(-1), (grad * nrm[:, None, :]).sum(-1)
                    mf[:, :, u] += (wa[..., None] * (fg[..., None] * nrm[:, None, :] - f * ng[..., None])).sum(1)
        self.lam, self.mf = lam, mf

    @staticmethod
    def _green(d):
        r = H * d.square().sum(-1).to(F64).sqrt()
        far = torch.where(r == 0.0, 1.0, r)
        return torch.where(r == 0.0, 0.0, torch.exp(-1j * K * far) / (4.0 * math.pi * far))

    def _spectrum(self):
        self.L = [_smooth(2 * v - 1) for v in self.n]
        ax = []
        for n, L in zip(self.n, self.L):
            i = torch.arange(L, device=DEV)
            ax.append((torch.where(i < n, i, torch.where(i > L - n, i - L, 1 << 20))))
        d = torch.stack(torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij"), -1)
        here = (d < (1 << 20)).all(-1)
        self.ghat = torch.fft.fftn(torch.where(here, self._green(torch.where(here[..., None], d, 0)), 0.0))

    def _pairs(self):
        """All (m, n) with |c_m - c_n| <= 3 h, row by row: candidates from the 27 cells around each centre."""
        r = 3.0 * H
        c = self.centre
        cell = torch.floor((c - c.amin(0)) / (r * 1.0001)).long()
        dims = (cell.amax(0) + 3).tolist()
        at = lambda v: (v[:, 2] * dims[1] + v[:, 1]) * dims[0] + v[:, 0]  # noqa: E731
        code, order = torch.sort(at(cell + 1))
        rows, cols = [], []
        for dz in (0, 1, 2):
            for dy in (0, 1, 2):
                for dx in (0, 1, 2):
                    want = at(cell + torch.tensor([dx, dy, dz], device=DEV))
                    a, b = torch.searchsorted(code, want), torch.searchsorted(code, want, right=True)
                    count = b - a
                    m = torch.repeat_interleave(torch.arange(self.N, device=DEV), count)
                    first = torch.repeat_interleave(torch.cumsum(count, 0) - count - a, count)
                    n = order[torch.arange(len(m), device=DEV) - first]
                    d = c[m] - c[n]
                    ok = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2] <= r * r
                    rows.append(m[ok])
                    cols.append(n[ok])
        key, _ = torch.sort(torch.cat(rows) * self.N + torch.cat(cols))
        return key // self.N, key % self.N

    def _blocks(self, P, Q, touch):
        """For test triangles P and sources Q (all touching or none): EFIE blocks [K, 3, 3], and MFIE ones for a CFIE."""
        bt, wt = _rule(5 if touch else 3)
        bs, ws = _rule(4)
        pv, qv, ap, aq = self.tv[P], self.tv[Q], self.area[P], self.area[Q]
        rt, rs = torch.einsum("qv,nvx->nqx", bt, pv), torch.einsum("qv,nvx->nqx", bs, qv)
        D = rt[:, :, None] - rs[:, None]
        R = D.square().sum(-1).sqrt()
        w = (ap * aq)[:, None, None] * wt[:, None] * ws
        if touch:  # (exp(-jkR) - 1) / (4 pi R); the rest in closed form below
            x = 0.5 * K * R
            G = (-1j * K / (4.0 * math.pi)) * torch.where(x == 0, 1.0, torch.sin(x) / torch.where(x == 0, 1.0, x)) * torch.exp(-1j * x)
        else:
            G = torch.exp(-1j * K * R) / (4.0 * math.pi * R)
        Gw = G * w
        ra, rb = rt[:, :, None] - pv[:, None], rs[:, :, None] - qv[:, None]  # [K, q, slot, 3]
        T = torch.einsum("kij,kiax,kjbx->kab", Gw, ra.to(C128), rb.to(C128)) / 4.0
        T -= (Gw.sum((1, 2)) / (K * K))[:, None, None]
        if touch:
            nt = rt.shape[1]
            one = torch.zeros((len(P), nt), dtype=F64, device=DEV)
            vec = torch.zeros((len(P), nt, 3), dtype=F64, device=DEV)
            nh = self.normal[Q][:, None]
            h = ((rt - qv[:, None, 0]) * nh).sum(-1)
            rho = rt - h[..., None] * nh
            for i in range(3):  # int 1/R and int (rho' - rho)/R over the source triangle, edge by edge
                a, b = qv[:, i], qv[:, (i + 1) % 3]
                e = b - a
                el = e.square().sum(-1).sqrt()
                along = e / el[:, None]
                out = torch.linalg.cross(along, self.normal[Q])
                lp = ((b[:, None] - rho) * along[:, None]).sum(-1)
                lm = ((a[:, None] - rho) * along[:, None]).sum(-1)
                t = ((a[:, None] - rho) * out[:, None]).sum(-1)
                r2 = t * t + h * h
                rp, rm = (r2 + lp * lp).sqrt(), (r2 + lm * lm).sqrt()
                ok = r2 > 1e-30 * (el * el)[:, None]
                r2s = torch.where(ok, r2, 1.0)
                num = torch.where(lp >= 0, rp + lp, r2s / (rp - lp))
                den = torch.where(lm >= 0, rm + lm, r2s / (rm - lm))
                f = torch.where(ok, torch.log(num / den), 0.0)
                ang = torch.atan(t * lp / (r2s + h.abs() * rp)) - torch.atan(t * lm / (r2s + h.abs() * rm))
                one += torch.where(ok, t * f - h.abs() * ang, 0.0)
                vec += 0.5 * out[:, None] * (torch.where(ok, r2 * f, 0.0) + lp * rp - lm * rm)[..., None]
            wp = ap[:, None] * wt / (4.0 * math.pi)
            V = vec[:, :, None] + (rho[:, :, None] - qv[:, None]) * one[..., None, None]
            T += torch.einsum("ki,kiax,kibx->kab", wp, ra, V) / 4.0 - ((wp * one).sum(1) / (K * K))[:, None, None]
        T /= (ap * aq)[:, None, None]
        if self.alpha == 1.0:
            return T, None
        nP = self.normal[P]
        flat = (torch.linalg.cross(nP, self.normal[Q]).abs().amax(-1) == 0) & (((qv[:, 0] - pv[:, 0]) * nP).sum(-1).abs() == 0)
        flat |= P == Q
        Rs = torch.where(flat[:, None, None], 1.0, R)
        gw = -(1.0 + 1j * K * Rs) * torch.exp(-1j * K * Rs) / (4.0 * math.pi * Rs ** 3) * w
        gw = torch.where(flat[:, None, None], 0.0, gw)
        aD = torch.einsum("kiax,kijx->kija", ra, D).to(C128)
        nb = torch.einsum("kx,kjbx->kjb", nP, rb).to(C128)
        nD = torch.einsum("kx,kijx->kij", nP, D)
        B = torch.einsum("kij,kija,kjb->kab", gw, aD, nb) - torch.einsum("kij,kiax,kjbx->kab", gw * nD, ra.to(C128), rb.to(C128))
        B /= (4.0 * ap * aq)[:, None, None]
        b3, w3 = _rule(3)
        r3 = torch.einsum("qv,nvx->nqx", b3, pv)[:, :, None] - pv[:, None]
        gram = torch.einsum("i,kiax,kibx->kab", w3, r3, r3) / (4.0 * ap)[:, None, None]
        return T, 0.5 * torch.where((P == Q)[:, None, None], gram, 0.0) - B

    def _near(self):
        rows, cols = self._pairs()
        nt = len(self.tris)
        combos = [(tm[rows] * nt + tn[cols], sm[rows] * 3 + sn[cols], gm * gn)
                  for tm, sm, gm in self.half for tn, sn, gn in self.half]
        keys = torch.cat([torch.unique(k) for k, _, _ in combos])
        keys = torch.unique(torch.cat([keys, (keys % nt) * nt + keys // nt]))
        P, Q = keys // nt, keys % nt
        touch = (self.tris[P][:, :, None] == self.tris[Q][:, None, :]).any(-1).any(-1)
        T = torch.empty((len(keys), 9), dtype=C128, device=DEV)
        B = torch.empty((len(keys), 9), dtype=C128, device=DEV) if self.alpha != 1.0 else None
        for sing in (False, True):
            which = torch.nonzero(touch == sing)[:, 0]
            for s in range(0, len(which), 1 << 17):
                at = which[s:s + (1 << 17)]
                t, b = self._blocks(P[at], Q[at], sing)
                T[at] = t.reshape(-1, 9)
                if B is not None:
                    B[at] = b.reshape(-1, 9)
        z = torch.zeros(len(rows), dtype=C128, device=DEV)
        zm = torch.zeros_like(z)
        turned = lambda s: (s % 3) * 3 + s // 3  # noqa: E731
        for key, slots, sign in combos:
            i, j = torch.searchsorted(keys, key), torch.searchsorted(keys, (key % nt) * nt + key // nt)
            z += 0.5 * sign * (T[i, slots] + T[j, turned(slots)])
            if B is not None:
                zm += sign * B[i, slots]
        ll = self.length[rows] * self.length[cols]
        z *= 1j * K * ETA0 * ll
        zm *= ll
        # minus what the grid gives for the same pairs, by the offset between the two stencils
        d = self.anc[rows] - self.anc[cols]
        span = 64
        code, back = torch.unique(((d[:, 2] + span) * 2 * span + d[:, 1] + span) * 2 * span + d[:, 0] + span, return_inverse=True)
        order = torch.argsort(back, stable=True)
        start = torch.searchsorted(back[order], torch.arange(len(code) + 1, device=DEV)).tolist()
        fac = torch.tensor([1.0, 1.0, 1.0, -1.0 / (K * K)], dtype=F64, device=DEV)
        for q in range(len(code)):
            for s in range(start[q], start[q + 1], 1 << 18):
                at = order[s:min(start[q + 1], s + (1 << 18))]
                G = self._green(d[at[0]] + self.off[:, None] - self.off[None])
                ln = self.lam[cols[at]]
                for part, unit in ((G.real, 1.0), (G.imag, 1j)):
                    pot = ln @ part.T.contiguous()  # potentials of n's stencil at m's nodes
                    z[at] -= unit * 1j * K * ETA0 * ((self.lam[rows[at]] * pot).sum(-1) * fac).sum(-1)
                    if B is not None:
                        zm[at] += unit * (self.mf[rows[at]] * pot[:, :3]).sum((-1, -2))
        val = z if B is None else self.alpha * z + (1.0 - self.alpha) * ETA0 * zm
        self.near = torch.sparse_coo_tensor(torch.stack([rows, cols]), val, (self.N, self.N)).coalesce().to_sparse_csr()
        diag = torch.zeros(self.N, dtype=C128, device=DEV)
        own = rows == cols
        diag[rows[own]] = val[own]
        self.diag = diag

    def product(self, x):
        out = []
        nx, ny, nz = self.n
        lam = self.lam.permute(1, 0, 2)  # [4, N, S]
        fac = 1j * K * ETA0 * torch.tensor([1.0, 1.0, 1.0, -1.0 / (K * K)], dtype=F64, device=DEV)
        for v in x:
            q = torch.zeros((4, nz * ny * nx), dtype=C128, device=DEV)
            for c in range(4):
                src = (lam[c] * v[:, None]).ravel()
                q[c].real.index_add_(0, self.node.ravel(), src.real)
                q[c].imag.index_add_(0, self.node.ravel(), src.imag)
            y = self.near @ v
            for c in range(4):
                phi = torch.fft.ifftn(torch.fft.fftn(q[c].reshape(nz, ny, nx), s=self.L[::-1]) * self.ghat)
                phi = phi[:nz, :ny, :nx].ravel()[self.node]
                y += self.alpha * fac[c] * (lam[c] * phi).sum(-1)
                if self.alpha != 1.0 and c < 3:
                    y -= (1.0 - self.alpha) * ETA0 * (self.mf[:, c] * phi).sum(-1)
            out.append(y)
        return torch.stack(out)

    def waves(self, k, p):
        V = torch.zeros((len(k), self.N), dtype=C128, device=DEV)
        for tri, _sign, _area, pts, f, wa in self._halves(4):
            for b in range(len(k)):
                kk, pp = torch.tensor(k[b], device=DEV), torch.tensor(p[b], device=DEV)
                field = self.alpha * pp + (1.0 - self.alpha) * torch.linalg.cross(
                    self.normal[tri], torch.linalg.cross(kk, pp).expand(self.N, 3))
                V[b] += ((f * field[:, None, :]).sum(-1) * torch.exp(-1j * K * (pts @ kk)) * wa).sum(-1)
        return V

    def solve(self, V, tol=1e-13, m=150):
        """Diagonally preconditioned GMRES of one right-hand side at a time, modified Gram-Schmidt."""
        X = torch.zeros_like(V)
        for b in range(len(V)):
            for _ in range(6):
                r = V[b] - self.product(X[b][None])[0]
                beta = torch.linalg.norm(r)
                if beta <= tol * torch.linalg.norm(V[b]):
                    break
                basis, Hm = [r / beta], torch.zeros((m + 1, m), dtype=C128, device=DEV)
                for j in range(m):
                    w = self.product((basis[j] / self.diag)[None])[0]
                    for _again in range(2):
                        for i in range(j + 1):
                            hij = torch.vdot(basis[i], w)
                            Hm[i, j] += hij
                            w = w - hij * basis[i]
                    Hm[j + 1, j] = torch.linalg.norm(w)
                    basis.append(w / Hm[j + 1, j])
                    if j % 10 == 9 or j == m - 1:
                        rhs = torch.zeros(j + 2, dtype=C128, device=DEV)
                        rhs[0] = beta
                        A = Hm[:j + 2, :j + 1]
                        y = torch.linalg.lstsq(A, rhs[:, None]).solution[:, 0]
                        if torch.linalg.norm(A @ y - rhs) <= 0.1 * tol * torch.linalg.norm(V[b]):
                            break
                X[b] += (torch.stack(basis[:len(y)], 1) @ y) / self.diag
        return X

    def pattern(self, X, theta, phi):
        th, ph = torch.tensor(theta, device=DEV), torch.tensor(phi, device=DEV)
        st, ct, sp, cp = th.sin(), th.cos(), ph.sin(), ph.cos()
        out = torch.stack([st * cp, st * sp, ct], 1)
        far = torch.zeros((len(X), len(th), 3), dtype=C128, device=DEV)
        for _tri, _sign, _area, pts, f, wa in self._halves(3):
            cur = torch.einsum("bn,nqx,nq->bnqx", X, f.to(C128), wa.to(C128)).reshape(len(X), -1, 3)
            flat = pts.reshape(-1, 3)
            for s in range(0, len(flat), 1 << 15):
                wave = torch.exp(1j * K * (out @ flat[s:s + (1 << 15)].T))
                far += torch.einsum("dp,bpx->bdx", wave, cur[:, s:s + (1 << 15)])
        scale = K * K * ETA0 * ETA0 / (4.0 * math.pi)
        up = torch.stack([ct * cp, ct * sp, -st], 1).to(C128)
        across = torch.stack([-sp, cp, torch.zeros_like(sp)], 1).to(C128)
        return [(scale * (far * v).sum(-1).abs().square()).cpu().numpy() for v in (up, across)]


def exact(case, seed):
    bodies = _meshes(case)
    if sum(len(t) for _, t in bodies) * (2 if case["cfie"] else 1) > 420_000 or case["op"] == "solve" and case["size"] > 2.2:
        return None  # too long: the near entries of a large body, or its many products
    n = case["nrhs"]
    if case["op"] == "rcs":
        a = _Exact.__new__(_Exact)
        a._near = a._spectrum = a._weights = lambda: None
        a.__init__(*bodies[0], 1.0)
        return a.pattern(_vector(n, a.N, seed, C128), *_directions(case))
    ops = [_Exact(v, t, ALPHA if case["cfie"] else 1.0) for v, t in bodies]
    if case["op"] == "solve":
        return ops[0].solve(ops[0].waves(*_waves(n, seed)))
    if case["op"] != "pack":
        return ops[0].product(_vector(n, ops[0].N, seed, _dtype(case)).to(C128))
    y = torch.zeros((n * len(ops), max(o.N for o in ops)), dtype=C128, device=DEV)
    for i, o in enumerate(ops):
        y[i * n:(i + 1) * n, :o.N] = o.product(_vector(n, o.N, seed * 16 + i, torch.complex64).to(C128))
    return y
