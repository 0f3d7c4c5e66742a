"""What is timed: the work that a user of the fast EFIE has it do.

A case names a body (a geodesic sphere of `freq`, an ellipsoid, or a finely and
a coarsely meshed sphere side by side), the method's parameters and one call:

  matvec  y = T x for `nrhs` device vectors (the product inside a Krylov solve)
  host    the same product on pinned host vectors (copies included)
  rhs     `nrhs` plane-wave right-hand sides
  solve   GMRES for `nrhs` plane waves to a 1e-6 true residual
  setup   a new geometry: setup, one product, teardown

Lengths are in wavelengths (k = 2 pi).  The mesh edge is `edge` times about 1.1,
the leaf grid spacing is 0.1, as in the bench's workloads.
"""
import functools
import math

import numpy as np
import torch

import paper_2606_13482_gb300 as G

K = 2 * math.pi
SPACING = 0.1


def _case(name, call, **kw):
    c = dict(call=call, body="sphere", freq=8, edge=0.05, p=3, levels=2, precision="mixed", factorization="star",
             nrhs=1)
    c.update(kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest problem: a 1-wavelength sphere, one FP64 vector; launches and latency
        _case("small_fp64_1", "matvec", freq=8, edge=0.0625, precision="fp64"),
        # one iteration of a mixed solve with one right-hand side on a mid-size scatterer
        _case("iteration_mixed_1", "matvec", freq=15, levels=1),
        # a batched mixed solve's product: 4-wavelength sphere, 8 plane waves
        _case("sphere4_mixed_8", "matvec", freq=40, nrhs=8),
        # the plain FP64 form of the same product (reference solves, true residuals)
        _case("sphere4_fp64_8", "matvec", freq=40, nrhs=8, precision="fp64"),
        # a count of vectors that is no multiple of 8, splines of higher degree
        _case("ragged_p5_mixed_19", "matvec", freq=27, p=5, nrhs=19),
        # large scatterer, many incidences at once: throughput
        _case("sphere10_mixed_64", "matvec", freq=100, levels=3, nrhs=64),
        # vectors that live in host memory: copies overlap the products
        _case("sphere6_host_32", "host", freq=60, levels=3, nrhs=32),
        # uneven mesh on the nonuniform octree
        _case("uneven_tree_mixed_64", "matvec", body="uneven", freq=50, levels=0, nrhs=64),
        # the direct factorization, a pair of 8-vector chunks
        _case("direct_mixed_16", "matvec", freq=20, factorization="direct", nrhs=16),
        # monostatic sweep: excitations of 360 azimuth angles on an ellipsoid
        _case("planewaves_360", "rhs", body="ellipsoid", freq=44, nrhs=360),
        # whole solve of a small problem in the plain FP64 form
        _case("solve_fp64_2", "solve", freq=8, edge=0.0625, precision="fp64", nrhs=2),
        # a new geometry: setup (host plan, FP64 near-field assembly, kernel spectra) and its first product
        _case("setup_mixed_1", "setup", freq=20),
    ]


def _levels(freq, edge):
    depth = max(1, math.ceil(math.log2(2 * freq * edge / (4 * SPACING))))
    return min(3, max(1, depth - 1))


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    p = rng.choice([3, 3, 3, 1, 2, 4, 5, 6])
    kind = rng.choice(["mixed", "mixed", "mixed", "mixed", "fp64", "fp64", "host", "tree", "direct", "rhs", "solve",
                       "setup"])
    if kind == "rhs":
        return _case(None, "rhs", body="ellipsoid", freq=logint(8, 44), nrhs=logint(1, 360))
    if kind == "solve":
        f = rng.randint(6, 10)
        return _case(None, "solve", freq=f, levels=1, precision="fp64", nrhs=rng.randint(1, 4))
    if kind == "setup":
        f = logint(8, 24)
        return _case(None, "setup", freq=f, p=p, levels=_levels(f, 0.05),
                     precision=rng.choice(["mixed", "fp64"]))
    if kind == "tree":
        return _case(None, "matvec", body="uneven", freq=rng.randint(32, 50), levels=0, nrhs=logint(1, 64))
    if kind == "fp64":
        f = logint(8, 40)
        return _case(None, "matvec", freq=f, p=p, levels=_levels(f, 0.05), precision="fp64",
                     nrhs=logint(1, 8 if f > 20 else 32))
    if kind == "direct":
        f = logint(12, 40)
        return _case(None, "matvec", freq=f, p=p, levels=_levels(f, 0.05), factorization="direct", nrhs=logint(1, 64))
    f = logint(10, 80)
    return _case(None, "host" if kind == "host" else "matvec", body=rng.choice(["sphere", "ellipsoid"]), freq=f, p=p,
                 levels=_levels(f, 0.05), nrhs=logint(1, 64))


# ---------------------------------------------------------------- meshes
def _geodesic(freq):
    """Unit sphere: every icosahedron face split into freq^2 triangles."""
    t = (1 + math.sqrt(5)) / 2
    iv = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                   [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]]) / math.sqrt(1 + t * t)
    edge2 = ((iv[:, None] - iv[None]) ** 2).sum(-1)
    near = np.isclose(edge2, np.min(edge2[edge2 > 1e-9]))
    faces = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
             if near[a, b] and near[b, c] and near[a, c]]
    ij = [(i, j) for i in range(freq + 1) for j in range(freq + 1 - i)]
    at = {q: n for n, q in enumerate(ij)}
    tri = [(at[i, j], at[i + 1, j], at[i, j + 1]) for i, j in ij if i + j < freq]
    tri += [(at[i + 1, j], at[i + 1, j + 1], at[i, j + 1]) for i, j in ij if i + j + 1 < freq]
    w = np.array([(freq - i - j, i, j) for i, j in ij], dtype=np.float64) / freq
    pts = np.concatenate([w @ iv[list(f)] for f in faces])
    tris = np.concatenate([np.array(tri) + n * len(ij) for n in range(len(faces))])
    _, first, inv = np.unique(np.round(pts * (1 << 24)).astype(np.int64), axis=0, return_index=True,
                              return_inverse=True)
    V = pts[first]
    T = inv.reshape(-1)[tris].astype(np.int32)
    V = V / np.linalg.norm(V, axis=1, keepdims=True)
    a, b, c = V[T[:, 0]], V[T[:, 1]], V[T[:, 2]]
    flip = np.einsum("ij,ij->i", np.cross(b - a, c - a), a + b + c) < 0
    T[flip] = T[flip][:, [0, 2, 1]]
    return V, T


def _mesh(c):
    f = c["freq"]
    if c["body"] == "uneven":
        # a finely meshed sphere beside a coarsely meshed one, 2.5 : 1 in radius
        g = max(6, round(0.28 * f))
        (Va, Ta), (Vb, Tb) = _geodesic(f), _geodesic(g)
        ra, rb = 0.02 * f, 2.5 * 0.02 * f
        x = (ra + rb + 0.02 * f) / 2
        return (np.concatenate([Va * ra + [-x, 0.0, 0.0], Vb * rb + [x, 0.1, 0.05]]),
                np.concatenate([Ta, Tb + len(Va)]).astype(np.int32))
    V, T = _geodesic(f)
    axes = np.array([1.0, 0.8, 0.65] if c["body"] == "ellipsoid" else [1.0, 1.0, 1.0])
    return V * (axes * f * c["edge"]), T


# ---------------------------------------------------------------- handles
_FACT = {"star": 0, "direct": 1}


def _setup(c, mesh):
    kw = dict(precision=G.EFIE_FP64 if c["precision"] == "fp64" else G.EFIE_MIXED,
              factorization=_FACT[c["factorization"]])
    if c["body"] == "uneven":
        return G.EFIE(*mesh, K, c["p"], tree=dict(max_elems=200, max_prot=0.25, top=2), **kw)
    return G.EFIE(*mesh, K, c["p"], SPACING, c["levels"], **kw)


_kept = {}


def _handle(c):
    """The handle that a program keeps for its geometry, whatever its vectors; one at a time."""
    key = tuple(sorted((k, v) for k, v in c.items() if k not in ("name", "call", "nrhs")))
    if key not in _kept:
        _kept.clear()
        _kept[key] = _setup(c, _mesh(c))
    return _kept[key]


def _waves(nrhs, seed):
    rng = np.random.default_rng(seed)
    phi = 2 * np.pi * (np.arange(nrhs) + rng.random()) / nrhs
    khat = np.stack([-np.cos(phi), -np.sin(phi), np.zeros(nrhs)], 1)
    return khat, np.tile([0.0, 0.0, 1.0], (nrhs, 1))


def _vectors(c, seed, h):
    """Unit vectors as a Krylov solve holds them: plane-wave excitations (the
    first basis vectors) and, for every other one, a noisy current."""
    n = c["nrhs"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = h.rhs_planewave(*_waves(n, seed))
    z = torch.view_as_complex(torch.randn((n, h.N, 2), dtype=torch.float64, device="cuda", generator=gen))
    x /= x.norm(dim=1, keepdim=True)
    z /= z.norm(dim=1, keepdim=True)
    x[::2] += z[::2]
    x[1::2] += 0.05 * z[1::2]
    return x


def prepare(case, seed):
    c = case
    if c["call"] == "setup":
        mesh = _mesh(c)
        N = 3 * len(mesh[1]) // 2
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.view_as_complex(torch.randn((c["nrhs"], N, 2), dtype=torch.float64, device="cuda", generator=gen))
        return dict(c=c, mesh=mesh, x=x)
    h = _handle(c)
    s = dict(c=c, h=h)
    if c["call"] == "rhs":
        s["waves"] = _waves(c["nrhs"], seed)
    elif c["call"] == "solve":
        s["x"] = h.rhs_planewave(*_waves(c["nrhs"], seed))
        s["y"] = torch.empty_like(s["x"])
    else:
        s["x"] = _vectors(c, seed, h)
        if c["call"] == "host":
            s["x"] = s["x"].cpu().pin_memory()
            s["y"] = torch.empty_like(s["x"], pin_memory=True)
        else:
            s["y"] = torch.empty_like(s["x"])
    return s


def run(state):
    c = state["c"]
    if c["call"] == "setup":
        h = _setup(c, state["mesh"])
        y = h.matvec(state["x"])
        h.close()
        return y
    h = state["h"]
    if c["call"] == "rhs":
        return h.rhs_planewave(*state["waves"])
    if c["call"] == "solve":
        x, info, rc = h.solve(state["x"], tol=1e-6, x=state["y"])
        return x
    if c["call"] == "host":
        return h.matvec_host(state["x"], state["y"])
    return h.matvec(state["x"], state["y"])


# ---------------------------------------------------------------- work
@functools.lru_cache(maxsize=64)
def _counts(key):
    """(unknowns, triangles, near entries, per level (boxes, far pairs, offsets, n)) of a case's plan."""
    c = dict(key)
    mesh = _mesh(c)
    N, nt = 3 * len(mesh[1]) // 2, len(mesh[1])
    if c["body"] == "uneven":
        lv, nr, ntr = G.plan_adaptive(*mesh, K, c["p"])
        return N, nt, nr + ntr, [(x["n_boxes"], x["n_far_pairs"], 0, 2 * x["shat"] - 1) for x in lv]
    o = G.Options()
    o.factorization = _FACT[c["factorization"]]
    i, lv = G.plan(*mesh, K, c["p"], SPACING, c["levels"], o)
    return (N, nt, i["near_nnz_A"] + i["near_nnz_V"],
            [(x["n_boxes"], x["n_far_pairs"], x["n_offsets"], x["nfft"]) for x in lv])


def work(case):
    N, nt, near, levels = _counts(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "nrhs"))))
    R, call = case["nrhs"], case["call"]
    if call == "rhs":  # 36 points a triangle and wave: phase, sine and cosine, five sums
        return {"bytes": 16.0 * N * R + 24.0 * nt, "flops": 36.0 * 20 * nt * R}
    vb = 16 if case["precision"] == "fp64" else 8
    # a product: near entries and kernel spectra read once, vectors read and written; one complex
    # multiply-add per near entry and vector and per far pair, frequency and channel; the FFTs
    bytes_ = 16.0 * near + sum(vb * o * n ** 3 for _, _, o, n in levels) + 32.0 * N * R
    flops = 8.0 * near * R + sum(4.0 * R * (8.0 * q * n ** 3 + 2 * 5.0 * b * n ** 3 * math.log2(n ** 3))
                                 for b, q, _, n in levels if q)
    if call == "solve":  # a handful of Krylov steps is the least that reaches 1e-6
        return {"bytes": 10 * bytes_, "flops": 10 * flops}
    if call == "setup":  # 81 point pairs for every near pair of triangles, half of them by symmetry
        return {"bytes": bytes_ + 16.0 * near, "flops": flops + 0.5 * near / 3.25 * 81 * 20}
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64-bit values
# The Galerkin EFIE with RWG functions, written out densely in 64 bits: products are
# summed over all triangle pairs.  Quadrature: collapsed Gauss rules of 3 x 3 points on
# both triangles of a regular pair; for a close pair (centroids closer than two longest
# edges) a 4 x 4 rule outside, the static part inside in closed form (Wilton et al.
# 1984) and the remainder by a 4 x 4 rule, averaged over both orders of the pair.
def _rule(n):
    x, w = np.polynomial.legendre.leggauss(n)
    x, w = (x + 1) / 2, w / 2
    u, v = np.meshgrid(x, x, indexing="ij")
    return u.ravel(), (v * (1 - u)).ravel(), (np.outer(w, w) * (1 - u)).ravel()


class _Dense:
    def __init__(self, mesh, dev):
        V, T = mesh
        self.nt, self.dev = len(T), dev
        e = np.concatenate([T[:, [a, (a + 1) % 3]] for a in range(3)]).astype(np.int64)
        tri = np.tile(np.arange(self.nt), 3)
        opp = np.concatenate([T[:, (a + 2) % 3] for a in range(3)])
        up = e[:, 0] < e[:, 1]  # the edge runs upwards in this triangle: its c+
        order = np.lexsort((~up, e.max(1), e.min(1)))
        self.N = len(order) // 2
        side = order.reshape(self.N, 2)
        self.tri = torch.from_numpy(tri[side]).to(dev)
        free = opp[side]
        loc = np.argmax(T[tri[side]] == free[..., None], axis=2)
        self.loc = torch.from_numpy(loc).to(dev)
        self.v = torch.from_numpy(V[T]).to(dev)
        e1, e2 = self.v[:, 1] - self.v[:, 0], self.v[:, 2] - self.v[:, 0]
        self.two_a = torch.linalg.cross(e1, e2).norm(dim=1)
        self.cen = self.v.mean(1)
        self.emax2 = (self.v - self.v.roll(-1, 1)).square().sum(2).amax(1)
        self.sign = torch.tensor([1.0, -1.0], dtype=torch.float64, device=dev)

    def points(self, t, n):
        xi, eta, w = (torch.from_numpy(a).to(self.dev) for a in _rule(n))
        v = self.v[t]
        e1, e2 = v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
        x = v[:, None, 0] + xi[:, None] * e1[:, None] + eta[:, None] * e2[:, None]
        return x, self.two_a[t][:, None] * w

    def regular(self, t, s):
        """I0 [t, s] and I[t, s, i, j] = int int (x - v_i).(y - v_j) g for all pairs of t and s."""
        X, wx = self.points(t, 3)
        Y, wy = self.points(s, 3)
        R = torch.cdist(X.reshape(-1, 3), Y.reshape(-1, 3), compute_mode="donot_use_mm_for_euclid_dist")
        R = R.view(len(t), 9, len(s), 9).clamp_min(1e-300)
        g = torch.polar(1 / (4 * math.pi * R), -K * R) * (wx[:, :, None, None] * wy[None, None])
        del R
        Xc, Yc = (a.to(torch.complex128) for a in (X - self.cen[t][:, None], Y - self.cen[s][:, None]))
        gy = torch.einsum("aqbp,bpd->aqbd", g, Yc)
        g0 = g.sum(3)
        I0, Ix, Iy = g0.sum(1), torch.einsum("aqb,aqd->abd", g0, Xc), gy.sum(1)
        Ixy = torch.einsum("aqbd,aqd->ab", gy, Xc)
        a = (self.v[t] - self.cen[t][:, None]).to(torch.complex128)
        b = (self.v[s] - self.cen[s][:, None]).to(torch.complex128)
        out = Ixy[:, :, None, None] - torch.einsum("aid,abd->abi", a, Iy)[:, :, :, None]
        out = out - torch.einsum("bjd,abd->abj", b, Ix)[:, :, None, :]
        return I0, out + torch.einsum("aid,bjd->abij", a, b) * I0[:, :, None, None]

    def static(self, r, v):
        """int 1/R and int (r' - rho)/R over the triangles v [P,3,3] at r [P,Q,3]; rho is r's foot."""
        n = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
        n = (n / n.norm(dim=1, keepdim=True))[:, None]
        d = ((r - v[:, None, 0]) * n).sum(-1)
        rho = r - d[..., None] * n
        one, vec = torch.zeros_like(d), torch.zeros_like(r)
        for i in range(3):
            a, b = v[:, None, i], v[:, None, (i + 1) % 3]
            t = (b - a) / (b - a).norm(dim=-1, keepdim=True)
            u = torch.linalg.cross(t.expand_as(n), n)
            lm, lp, p0 = ((a - rho) * t).sum(-1), ((b - rho) * t).sum(-1), ((a - rho) * u).sum(-1)
            q = p0 * p0 + d * d
            rm, rp = (r - a).norm(dim=-1), (r - b).norm(dim=-1)
            up = torch.where(lp >= 0, rp + lp, q / (rp - lp).clamp_min(1e-300))
            dn = torch.where(lm >= 0, rm + lm, q / (rm - lm).clamp_min(1e-300))
            lg = torch.where((up > 0) & (dn > 0), torch.log(up / dn), torch.zeros_like(q))
            at = torch.atan2(p0 * lp, q + d.abs() * rp) - torch.atan2(p0 * lm, q + d.abs() * rm)
            one += torch.where(p0.abs() > 1e-300, p0 * lg - d.abs() * at, torch.zeros_like(q))
            vec += (0.5 * (q * lg + lp * rp - lm * rm))[..., None] * u
        return one, vec, rho

    def close_one(self, t, s):
        """The close rule for pairs (t[p], s[p]), outside on t."""
        X, wx = self.points(t, 4)
        Y, wy = self.points(s, 4)
        one, vec, rho = self.static(X, self.v[s])
        R = (X[:, :, None] - Y[:, None]).norm(dim=-1)
        Rs = R.clamp_min(1e-300)
        rem = torch.complex(-2 * torch.sin(0.5 * K * R).square() / Rs,
                            -torch.where(R > 0, torch.sin(K * R) / Rs, torch.full_like(R, K)))
        rem = rem * (wy[:, None] / (4 * math.pi))
        cs = self.cen[s][:, None]
        i0 = one / (4 * math.pi) + rem.sum(2)
        iy = (vec + (rho - cs) * one[..., None]) / (4 * math.pi)
        iy = iy + torch.einsum("pab,pbd->pad", rem, (Y - cs).to(rem.dtype))
        b = (self.v[s] - cs).to(rem.dtype)
        inner = iy[:, None] - b[:, :, None] * i0[:, None, :, None]
        xv = (X[:, None] - self.v[t][:, :, None]).to(rem.dtype)
        wc = wx.to(rem.dtype)
        return (wc * i0).sum(1), torch.einsum("pq,piqd,pjqd->pij", wc, xv, inner)

    def pairs(self, t):
        """I0 [t, nt] and I [t, nt, 3, 3] of the triangles t with every triangle."""
        s = torch.arange(self.nt, device=self.dev)
        I0, I = self.regular(t, s)
        d2 = (self.cen[t][:, None] - self.cen[None]).square().sum(-1)
        a, b = torch.nonzero(d2 < 4 * torch.maximum(self.emax2[t][:, None], self.emax2[None]), as_tuple=True)
        for q in range(0, len(a), 4096):
            p, o = a[q:q + 4096], b[q:q + 4096]
            f0, f = self.close_one(t[p], o)
            g0, g = self.close_one(o, t[p])
            I0[p, o] = 0.5 * (f0 + g0)
            I[p, o] = 0.5 * (f + g.transpose(1, 2))
        return I0, I

    def apply(self, x):
        """T x for x [R, N]."""
        x = x.to(self.dev)
        R, cd = len(x), torch.complex128
        coef = (self.sign / self.two_a[self.tri]).to(cd)  # f = coef (x - v) on each side, div f = 2 coef
        src = torch.zeros((3 * self.nt, R), dtype=cd, device=self.dev)
        rho = torch.zeros((self.nt, R), dtype=cd, device=self.dev)
        for k in range(2):
            src.index_add_(0, 3 * self.tri[:, k] + self.loc[:, k], (coef[:, k] * x).T.contiguous())
            rho.index_add_(0, self.tri[:, k], (2 * coef[:, k] * x).T.contiguous())
        ya = torch.empty((3 * self.nt, R), dtype=cd, device=self.dev)
        yv = torch.empty((self.nt, R), dtype=cd, device=self.dev)
        m = max(1, min(64, 40_000 // self.nt))
        for q in range(0, self.nt, m):
            t = torch.arange(q, min(q + m, self.nt), device=self.dev)
            I0, I = self.pairs(t)
            yv[t] = I0 @ rho
            ya[3 * q:3 * q + 3 * len(t)] = I.permute(0, 2, 1, 3).reshape(3 * len(t), 3 * self.nt) @ src
        y = torch.zeros((R, self.N), dtype=cd, device=self.dev)
        for k in range(2):
            y += 1j * K * coef[:, k] * ya[3 * self.tri[:, k] + self.loc[:, k]].T
            y += 2 * coef[:, k] / (1j * K) * yv[self.tri[:, k]].T
        return y

    def waves(self, khat, pol):
        khat, pol = (torch.from_numpy(a).to(self.dev) for a in (khat, pol))
        X, w = self.points(torch.arange(self.nt, device=self.dev), 6)
        y = torch.empty((len(khat), self.N), dtype=torch.complex128, device=self.dev)
        for r in range(len(khat)):
            ph = torch.polar(w, -K * (X @ khat[r]))
            f0, f1 = ph.sum(1), (ph * (X @ pol[r])).sum(1)
            y[r] = 0
            for k in range(2):
                t = self.tri[:, k]
                v = self.v[t, self.loc[:, k]] @ pol[r]
                y[r] += self.sign[k] / self.two_a[t] * (f1[t] - v * f0[t])
        return y


def exact(case, seed):
    c, dev = case, "cuda" if torch.cuda.is_available() else "cpu"
    nt = 20 * c["freq"] ** 2
    if c["call"] == "rhs":
        return _Dense(_mesh(c), dev).waves(*_waves(c["nrhs"], seed))
    if c["body"] == "uneven" or nt > 8000:
        return None
    d = _Dense(_mesh(c), dev)
    if c["call"] == "solve":
        T = d.apply(torch.eye(d.N, dtype=torch.complex128))
        return torch.linalg.solve(T, d.waves(*_waves(c["nrhs"], seed)).T).T.contiguous()
    s = prepare(c, seed)
    return d.apply(s["x"])
