"""What users of this library have it do, as measurable cases.

Five kinds of calls, each through the public Python binding of the C ABI:

  build   steps 2 and 3 on a prepared partition, the library's main use: the local bases
          of every subdomain, the interface projection, the reduced solve, the lift.
  host    the same from host arrays, step 1 (the subdomain plan) included, and the
          solution read back: a program that solves one problem from end to end.
  wave    as build, on a streamed plan that works through the subdomains in waves.
  online  step 3 alone on bases that are kept: projection, reduced solve, lift and the
          energy norm of the result.
  solve   the allocation-free reduced solve on a caller's own block-sparse matrix, the
          call of a time-critical loop.

The sizes are those of the repository's workloads and of its scaling tests, or scaled
down from them where a pass would take longer than two seconds: cubes of Kuhn cells cut
into boxes or uneven Voronoi cells, subdomains extended by about half their width, ranks
8 to 64 with 5 to 10 extra sketch columns, lognormal coefficients, unit coefficients or
1e4-contrast spheres.  A case's seed gives the coefficient and the Gaussian sketch; the
mesh and the partition belong to the case.

Returned per case: the lifted solution on all nodes, the squared singular values of every
subdomain, the kept basis sizes and the reduced energy.  (Squared: the method computes
sigma^2, as eigenvalues with a normwise error; the roots of the trailing ones carry no
figures.)  Q_i and the reduced matrix are fixed only up to the signs of eigenvectors, so
the lifted solution stands for them.
"""
from __future__ import annotations

import ctypes
import functools
import itertools
import math

import numpy as np
import torch

from paper_2404_06260_gb300 import mor

# ------------------------------------------------------------------ the cases


def _case(name, kind, n, parts, r_hops, rank, oversample, precision, **kw):
    c = dict(name=name, kind=kind, n=n, parts=parts, partition="box", jitter=0.0,
             r_hops=r_hops, rank=rank, rank_hi=rank, oversample=oversample,
             precision=precision, field="lognormal", cg_rtol=1e-9, eps=0.0, sketch_div=0,
             sketch="field", explicit=False, wave=0)
    c.update(kw)
    return c


def listed():
    return [
        # the reduced solve of a small partition, called in a loop: launch latency
        dict(name="solve_27x12", kind="solve", grid=3, kq=12),
        # the same for some hundred subdomains: the block-sparse products count
        dict(name="solve_512x36", kind="solve", grid=8, kq=36),
        # step 3 on the bases of the smallest workload, binary64
        _case("online16", "online", 16, 2, 4, 8, 5, "fp64", cg_rtol=1e-12),
        # step 3 on many subdomains
        _case("online56", "online", 56, 7, 4, 24, 8, "mixed"),
        # the smallest workload (16^3 cells, 8 subdomains) in both precisions, the local
        # solves to ten figures
        _case("build16", "build", 16, 2, 4, 8, 5, "mixed", cg_rtol=1e-10),
        _case("build16_fp64", "build", 16, 2, 4, 8, 5, "fp64", cg_rtol=1e-10),
        # the benchmark's workload: 64^3 cells, 64 subdomains, rank 32 + 10
        _case("build64", "build", 64, 4, 8, 32, 10, "mixed"),
        # the binary64 path at a ragged size (45 cells in 3 boxes, 31 + 1 columns)
        _case("build45_fp64", "build", 45, 3, 7, 24, 7, "fp64", cg_rtol=1e-10),
        # an uneven batch: jittered mesh, Voronoi subdomains, ranks 16..64 per subdomain
        _case("uneven48", "build", 48, 40, -1, 16, 10, "mixed", partition="voronoi",
              jitter=0.2, rank_hi=64),
        # the scaling tests' sketch size, floor(|B| / 8) columns, kept by tolerance
        _case("wide25", "build", 25, 14, 4, 8, 0, "mixed", partition="voronoi",
              field="ones", eps=1e-2, sketch_div=8),
        # the paper-literal weights: dense factors and the explicit weighted SVD
        _case("explicit9", "build", 9, 2, 2, 8, 5, "fp64", explicit=True, cg_rtol=1e-12),
        # end to end from host arrays: high contrast (1e4 spheres), tight local solves
        _case("host47_spheres", "host", 47, 3, 7, 40, 10, "mixed", field="spheres",
              cg_rtol=1e-11),
    ]


# (extended rows) x columns x cost of the precision: a draw costs no more than build64
_MOST = 64 * 27.8 ** 3 * 44


def _cost(c):
    if c["kind"] == "solve":
        return 0.0
    k = c["rank_hi"] + c["oversample"]
    if c["sketch_div"]:
        k = 6.0 * _width(c) ** 2 / c["sketch_div"]
    w = 4.0 if c["precision"] == "fp64" else 1.0
    if c["field"] == "spheres":
        w *= 3.0
    if c["explicit"] or c["sketch"] == "paper":
        w *= 3.0
    return _subdomains(c) * _width(c) ** 3 * (k + 1) * w


def _subdomains(c):
    return c["parts"] if c["partition"] == "voronoi" else c["parts"] ** 3


def _hops(c):
    own = c["n"] ** 3 / _subdomains(c)
    return c["r_hops"] if c["r_hops"] > 0 else max(1, int(own ** (1 / 3) / 2 + 0.5))


def _width(c):
    """Mean width, in nodes, of an extended subdomain (hops cut off at the cube)."""
    p = _subdomains(c) ** (1 / 3)
    return min(c["n"], c["n"] / p + 2 * (_hops(c) + 1) * (1 - 1 / p) + 1)


def draw(rng):
    while True:
        c = _draw(rng)
        if _cost(c) <= _MOST:
            return c


def _draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["build", "build", "build", "build", "host", "wave", "online", "solve"])
    if kind == "solve":
        c = dict(name="", kind="solve", grid=rng.randint(2, 8), kq=4 * rng.randint(2, 16))
        del c["name"]
        return c
    what = rng.choice(["mixed", "mixed", "fp64", "uneven", "spheres", "wide", "paper",
                       "explicit"]) if kind == "build" else rng.choice(["mixed", "fp64"])
    n = log_int(14, 64)
    parts = rng.randint(2, max(2, n // 8))
    kw = {}
    if what in ("uneven", "wide"):
        n = log_int(14, 48 if what == "uneven" else 26)
        parts = max(8, round(n ** 3 / rng.uniform(1000.0, 3500.0)))
        kw.update(partition="voronoi")
    if what == "uneven":
        kw.update(jitter=round(rng.uniform(0.0, 0.2), 3))
    if what in ("paper", "explicit"):
        n, parts = (rng.randint(10, 16), 2) if what == "paper" else (rng.randint(8, 9), 2)
    if kind == "online":
        n, parts = log_int(14, 56), 0
        parts = max(2, min(7, round(n / rng.uniform(7.0, 12.0))))
    rank, over = log_int(6, 48), rng.randint(4, 10)
    c = _case("", kind, n, parts, 1, rank, over, "fp64" if what in ("fp64", "paper", "explicit")
              else "mixed", **kw)
    del c["name"]
    own = n / _subdomains(c) ** (1 / 3)
    c["r_hops"] = max(2, min(9, int(own * rng.uniform(0.4, 0.6))))
    if what == "uneven":
        c.update(r_hops=-1, rank=min(rank, 16), rank_hi=min(rank, 16) + rng.randint(8, 48))
    elif what == "wide":
        c.update(field="ones", eps=1e-2, sketch_div=8, rank=8, rank_hi=8, oversample=0)
    elif what == "spheres":
        c.update(field="spheres", cg_rtol=1e-11)
    elif what == "paper":
        c.update(sketch="paper", cg_rtol=1e-12, rank=min(rank, 16), rank_hi=min(rank, 16))
    elif what == "explicit":
        c.update(explicit=True, cg_rtol=1e-12, rank=min(rank, 12), rank_hi=min(rank, 12))
    elif what == "fp64" or n < 24 or rng.random() < 0.5:
        c.update(cg_rtol=1e-10)
    if kind == "wave":
        c["wave"] = rng.randint(2, max(2, _subdomains(c) // 2))
    return c


# ------------------------------------------------------------------ inputs


@functools.lru_cache(maxsize=32)
def _geometry(n, jitter, partition, parts):
    """Kuhn mesh of the unit cube and a partition of its nodes: (xyz, tets, dirichlet,
    owner), host arrays."""
    g = np.arange(n + 1) / n
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    xyz = np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1)
    face = (np.arange(n + 1) % n) == 0
    fz, fy, fx = np.meshgrid(face, face, face, indexing="ij")
    dirichlet = (fx | fy | fz).ravel().astype(np.uint8)
    s = np.array([1, n + 1, (n + 1) ** 2])
    cz, cy, cx = np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij")
    corner = (cx * s[0] + cy * s[1] + cz * s[2]).ravel()
    tets = np.empty((n ** 3, 6, 4), np.int32)
    for t, (a, b, c) in enumerate(itertools.permutations(range(3))):
        odd = (a, b, c) in ((0, 2, 1), (1, 0, 2), (2, 1, 0))
        p1, p2, p3 = s[a], s[a] + s[b], s.sum()
        if odd:
            p1, p2 = p2, p1
        for v, off in enumerate((0, p1, p2, p3)):
            tets[:, t, v] = corner + off
    tets = tets.reshape(-1, 4)
    rng = np.random.default_rng(n * 1000 + parts)
    if jitter > 0.0:
        d = rng.uniform(-jitter / n, jitter / n, size=xyz.shape)
        xyz = xyz + np.where(dirichlet[:, None] != 0, 0.0, d)
    if partition == "box":
        i = np.arange(n + 1)
        a = np.minimum(parts - 1, i * parts // n)
        oz, oy, ox = np.meshgrid(a, a, a, indexing="ij")
        owner = (ox + parts * (oy + parts * oz)).ravel()
    else:
        cen = xyz[rng.choice(len(xyz), size=parts, replace=False)]
        for _ in range(8):
            owner = _nearest(xyz, cen)
            cnt = np.maximum(np.bincount(owner, minlength=parts), 1)
            cen = np.stack([np.bincount(owner, weights=xyz[:, q], minlength=parts) / cnt
                            for q in range(3)], axis=1)
        owner = _nearest(xyz, cen)
        _, owner = np.unique(owner, return_inverse=True)
    return (np.ascontiguousarray(xyz), np.ascontiguousarray(tets), dirichlet,
            owner.astype(np.int32).ravel())


def _nearest(xyz, cen):
    best, owner = np.full(len(xyz), np.inf), np.zeros(len(xyz), np.int64)
    for i, c in enumerate(cen):
        d = ((xyz - c) ** 2).sum(axis=1)
        near = d < best
        best[near], owner[near] = d[near], i
    return owner


@functools.lru_cache(maxsize=8)
def _geometry_dev(n, jitter, partition, parts):
    xyz, tets, _, _ = _geometry(n, jitter, partition, parts)
    return torch.as_tensor(xyz, device="cuda"), torch.as_tensor(tets, device="cuda")


def _geo_key(c):
    return c["n"], c["jitter"], c["partition"], c["parts"]


def _kappa(c, seed):
    """Element coefficient on the GPU."""
    xyz, tets = _geometry_dev(*_geo_key(c))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nt = tets.shape[0]
    if c["field"] == "ones":
        return torch.ones(nt, dtype=torch.float64, device="cuda")
    if c["field"] == "lognormal":
        return torch.exp(torch.randn(nt, dtype=torch.float64, device="cuda", generator=gen))
    # spheres of radius 3..6 cells, 1e4 inside, at least a tenth of the elements
    cen = xyz[tets.long()].mean(dim=1)
    rng = np.random.default_rng(seed)
    inside = torch.zeros(nt, dtype=torch.bool, device="cuda")
    while float(inside.double().mean()) < 0.1:
        p = torch.as_tensor(rng.uniform(0.0, 1.0, size=3), device="cuda")
        r = rng.uniform(3.0, 6.0) / c["n"]
        inside |= ((cen - p) ** 2).sum(dim=1) < r * r
    return torch.where(inside, 1e4, 1.0).double()


def _ranks(c):
    if c["rank_hi"] <= c["rank"]:
        return None
    n_sub = int(_geometry(*_geo_key(c))[3].max()) + 1
    return np.random.default_rng(c["n"]).integers(c["rank"], c["rank_hi"] + 1, size=n_sub)


def _opts(c, seed):
    kw = dict(rank=c["rank"], oversample=c["oversample"], seed=seed, eps=c["eps"],
              precision=c["precision"], sketch=c["sketch"], cg_rtol=c["cg_rtol"],
              sketch_div=c["sketch_div"], explicit_svd=1 if c["explicit"] else 0)
    ranks = _ranks(c)
    if ranks is not None:
        kw["ranks"] = ranks
    return mor.basis_opts(**kw)


class _Loop:
    """A caller's own reduced system: block rows over a grid^3 box of subdomains coupled
    to their 14 neighbours in a Kuhn mesh, unit diagonal blocks, CG in about 50 steps."""

    def __init__(self, grid, kq, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = grid ** 3
        half = [d for d in itertools.product((0, 1), repeat=3) if any(d)]
        pairs = []
        for z, y, x in itertools.product(range(grid), repeat=3):
            for d in half:
                if max(x + d[0], y + d[1], z + d[2]) < grid:
                    i = x + grid * (y + grid * z)
                    pairs.append((i, i + d[0] + grid * (d[1] + grid * d[2])))
        self.pairs, self.n_sub, self.kq = pairs, n, kq
        scale = 0.47 / math.sqrt(14.0 * kq)
        off = scale * torch.randn((len(pairs), kq, kq), dtype=torch.float64, device="cuda",
                                  generator=gen)
        self.blocks = torch.stack([off, off.transpose(1, 2)], dim=1).contiguous()
        rows = [[] for _ in range(n)]
        for p, (i, j) in enumerate(pairs):
            rows[i].append((j, 2 * p))
            rows[j].append((i, 2 * p + 1))
        ptr = np.cumsum([0] + [len(r) for r in rows])
        flat = [e for r in rows for e in sorted(r)]

        def dev(v):
            return torch.as_tensor(np.asarray(v, np.int32), device="cuda")

        self.ptr, self.sub, self.blk = dev(ptr), dev([e[0] for e in flat]), dev(
            [e[1] for e in flat])
        self.bt = torch.randn(n * kq, dtype=torch.float64, device="cuda", generator=gen)
        self.x = torch.empty(n * kq, dtype=torch.float64, device="cuda")


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "solve":
        s.loop = _Loop(case["grid"], case["kq"], seed)
        return s
    xyz, tets, dirichlet, owner = _geometry(*_geo_key(case))
    kappa = _kappa(case, seed)
    s.opts = _opts(case, seed)
    if case["kind"] == "host":
        pin = [torch.as_tensor(a).pin_memory() for a in (xyz, tets, kappa.cpu().numpy(),
                                                         dirichlet)]
        s.host = (*pin, owner)
        return s
    xyz_d, tets_d = _geometry_dev(*_geo_key(case))
    mesh = mor.Mesh.from_device(xyz_d, tets_d, kappa, tets, dirichlet)
    s.sd = mor.Subdomains(mesh, owner, case["r_hops"], wave=case["wave"])
    if case["kind"] == "online":
        s.bases = mor.Bases(s.sd, s.opts)
    return s


# ------------------------------------------------------------------ one pass


def run(s):
    kind = s.case["kind"]
    if kind == "solve":
        return _solve(s.loop)
    if kind == "online":
        x, info = mor.Reduced(s.sd, s.bases).solve()
        u = mor.lift(s.sd, s.bases, x)
        return dict(u=u, energy=info["energy"], norm=mor.energy_norm(s.sd, u))
    sd = s.sd if kind != "host" else mor.Subdomains.from_host(*s.host, s.case["r_hops"])
    b = mor.Bases(sd, s.opts)
    x, info = mor.Reduced(sd, b).solve()
    u = mor.lift(sd, b, x)
    return dict(u=u.cpu() if kind == "host" else u, sigma2=b.sigma() ** 2, kept=b.kept,
                energy=info["energy"])


def _solve(c):
    def p(t):
        return ctypes.c_void_p(t.data_ptr())

    info = mor.SolveInfo()
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = mor._lib.mor_solve_reduced_noalloc(c.n_sub, c.kq, p(c.ptr), p(c.sub), p(c.blk),
                                            p(c.blocks), p(c.bt), 1e-12, 20000, st, p(c.x),
                                            ctypes.byref(info))
    if rc != mor.MOR_OK:
        raise mor.MorError(rc, mor._lib.mor_last_error().decode())
    return dict(x=c.x, energy=info.energy)


# ------------------------------------------------------------------ what a pass needs


def work(case):
    """Each input read once, each output written once; the flops of one application of
    the operators per solved column and of the dense contractions."""
    if case["kind"] == "solve":
        g, kq = case["grid"], case["kq"]
        pairs = sum((g - a) * (g - b) * (g - c) for a, b, c in
                    itertools.product((0, 1), repeat=3) if a + b + c)
        return dict(bytes=16.0 * pairs * kq * kq + 16.0 * g ** 3 * kq,
                    flops=4.0 * pairs * kq * kq)
    n = case["n"]
    nn, nt, n_sub = (n + 1) ** 3, 6 * n ** 3, _subdomains(case)
    k = case["rank_hi"] + case["oversample"]
    if case["sketch_div"]:
        k = 6.0 * _width(case) ** 2 / case["sketch_div"]
    kq = case["rank_hi"] + 1
    if case["kind"] == "online":
        iface = 3.0 * nn * case["parts"] / n  # couplings across the subdomains' faces
        return dict(bytes=8.0 * nn * kq + 32.0 * nn + 24.0 * nt + 8.0 * nn,
                    flops=4.0 * iface * kq * kq + 2.0 * nn * kq)
    rows = n_sub * _width(case) ** 3
    return dict(bytes=25.0 * nn + 24.0 * nt + 8.0 * nn + 8.0 * n_sub * k,
                flops=4 * 2.0 * 15 * rows * k + 8.0 * nn * k * k)


# ------------------------------------------------------------------ 64-bit values


def exact(case, seed):
    if case["kind"] == "solve":
        return _exact_solve(_Loop(case["grid"], case["kq"], seed))
    if case["wave"] or _width(case) > 14 or _subdomains(case) > 30 or case["eps"] > 0.0:
        return None  # dense factors of larger subdomains take too long
    u, sigma2, kept, energy = _exact_method(case, seed)
    if case["kind"] == "online":
        return dict(u=u, energy=energy, norm=math.sqrt(energy))
    return dict(u=u, sigma2=sigma2, kept=kept, energy=energy)


def _exact_solve(c):
    n, k = c.n_sub, c.kq
    K = torch.zeros((n, k, n, k), dtype=torch.float64, device="cuda")
    for i in range(n):
        K[i, :, i, :] = torch.eye(k, dtype=torch.float64, device="cuda")
    for p, (i, j) in enumerate(c.pairs):
        K[i, :, j, :] = c.blocks[p, 0]
        K[j, :, i, :] = c.blocks[p, 1]
    L = torch.linalg.cholesky(K.view(n * k, n * k))
    x = torch.cholesky_solve(c.bt[:, None], L)[:, 0]
    return dict(x=x, energy=float(c.bt @ x))


def _normals(counter0, cols, sub, tag, seed):
    """The library's documented Gaussian draws: Philox-4x32-10 of (counter0, column, sub,
    tag), Box-Muller in binary32.  Four arrays len(counter0) x cols."""
    u32 = np.uint64(0xFFFFFFFF)
    c = [np.broadcast_to(np.asarray(v, np.uint64), (len(counter0), cols)) for v in
         (np.asarray(counter0)[:, None], np.arange(cols)[None, :], sub, tag)]
    key = [seed & 0xFFFFFFFF, seed >> 32]
    for _ in range(10):
        p, q = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(q >> np.uint64(32)) ^ c[1] ^ np.uint64(key[0]), q & u32,
             (p >> np.uint64(32)) ^ c[3] ^ np.uint64(key[1]), p & u32]
        key = [(key[0] + 0x9E3779B9) & 0xFFFFFFFF, (key[1] + 0xBB67AE85) & 0xFFFFFFFF]
    f = np.float32

    def series(coef, t):
        acc = np.full_like(t, f(coef[0]))
        for a in coef[1:]:
            acc = acc * t + f(a)
        return acc

    def unit(x):
        return ((x >> np.uint64(9)) * np.uint64(2) + np.uint64(1)).astype(f) * f(2.0 ** -24)

    def log(v):
        m, e = np.frexp(v)
        m, e = (m * f(2)).astype(f), e - 1
        high = m > f(math.sqrt(2.0))
        m, e = np.where(high, m * f(0.5), m), e + high
        s = (m - f(1)) / (m + f(1))
        return e.astype(f) * f(math.log(2.0)) + (s + s) * series(
            [1 / 9, 1 / 7, 1 / 5, 1 / 3, 1.0], s * s)

    def circle(v):
        t = v * f(8)
        q = np.floor(t)
        o = q.astype(np.int64)
        th = np.where(o & 1, f(1) - (t - q), t - q) * f(math.pi / 4)
        t2 = th * th
        sn = th + th * (series([1 / 362880, -1 / 5040, 1 / 120, -1 / 6], t2) * t2)
        cs = series([-1 / 3628800, 1 / 40320, -1 / 720, 1 / 24, -0.5, 1.0], t2)
        swap = np.isin(o, (1, 2, 5, 6))
        return (np.where(swap, sn, cs) * np.where((o >= 2) & (o <= 5), f(-1), f(1)),
                np.where(swap, cs, sn) * np.where(o >= 4, f(-1), f(1)))

    out = []
    for a, b in ((0, 1), (2, 3)):
        r = np.sqrt(f(-2) * log(unit(c[a])))
        cc, ss = circle(unit(c[b]))
        out += [r * cc, r * ss]
    return out


def _exact_method(case, seed):
    """The method on dense matrices in 64 bits: per subdomain the optimal local space from
    the sketch (or the explicit weighted SVD), then the Galerkin solution in their sum."""
    dev = dict(dtype=torch.float64, device="cuda")
    xyz, tets, dirichlet, owner = _geometry(*_geo_key(case))
    kap = _kappa(case, seed)
    T = torch.as_tensor(tets, device="cuda").long()
    own = torch.as_tensor(owner, device="cuda").long()
    free = torch.as_tensor(dirichlet, device="cuda") == 0
    nn, nt = len(xyz), len(tets)
    X = torch.as_tensor(xyz, device="cuda")[T]
    J = X[:, 1:] - X[:, :1]
    vol = torch.linalg.det(J) / 6.0
    G = torch.linalg.inv(J).transpose(1, 2)
    G = torch.cat([-G.sum(dim=1, keepdim=True), G], dim=1)
    Ke = (G @ G.transpose(1, 2)) * vol[:, None, None]
    He = Ke + (torch.ones(4, 4, **dev) + torch.eye(4, **dev)) * (vol / 20.0)[:, None, None]
    Ae = Ke * kap[:, None, None]
    Le = torch.linalg.cholesky(He)

    def assemble(E, t, dofs):
        loc = torch.full((nn,), -1, dtype=torch.long, device="cuda")
        loc[dofs] = torch.arange(len(dofs), device="cuda")
        r = loc[T[t]]
        i, j = r[:, :, None].expand(-1, 4, 4), r[:, None, :].expand(-1, 4, 4)
        ok = (i >= 0) & (j >= 0)
        M = torch.zeros(len(dofs) * len(dofs), **dev)
        M.index_add_(0, (i * len(dofs) + j)[ok], E[t][ok])
        return M.view(len(dofs), len(dofs))

    load = torch.zeros(nn, **dev).index_add_(0, T.reshape(-1),
                                             (vol / 4.0).repeat_interleave(4))
    deg = torch.bincount(T.reshape(-1), minlength=nn)
    ranks = _ranks(case)
    n_sub = int(own.max()) + 1
    widest = case["oversample"] + int(ranks.max() if ranks is not None else case["rank"])
    V, sig, kept = [], [], []
    for i in range(n_sub):
        mine = own == i
        m = int(ranks[i]) if ranks is not None else case["rank"]
        k = m + case["oversample"]
        hops = case["r_hops"] if case["r_hops"] > 0 else max(
            1, int(np.floor(np.cbrt(float(mine.sum())) / 2.0 + 0.5)))
        ball = mine.clone()
        for _ in range(hops):
            ball[T[ball[T].any(dim=1)].reshape(-1)] = True
        plus, omega = ball[T].any(dim=1), mine[T].any(dim=1)
        cnt = torch.bincount(T[plus].reshape(-1), minlength=nn)
        I = torch.nonzero((cnt == deg) & free)[:, 0]
        B = torch.nonzero((cnt > 0) & (cnt < deg) & free)[:, 0]
        seen = torch.zeros(nn, dtype=torch.bool, device="cuda")
        seen[T[omega].reshape(-1)] = True
        W = torch.nonzero(seen & free)[:, 0]
        nI, dofs = len(I), torch.cat([I, B])
        A, H = assemble(Ae, plus, dofs), assemble(He, plus, dofs)
        LA, LH = torch.linalg.cholesky(A[:nI, :nI]), torch.linalg.cholesky(H)
        Hw = assemble(He, omega, W)
        R = torch.linalg.cholesky(Hw).T
        at = torch.full((nn,), -1, dtype=torch.long, device="cuda")
        at[dofs] = torch.arange(len(dofs), device="cuda")
        w = at[W]
        u0 = torch.cholesky_solve(load[I][:, None], LA)
        if case["explicit"]:
            Z = torch.cholesky_solve(A[:nI, nI:], LA)[w]
            Rbb = LH[nI:, nI:].T
            Y = torch.linalg.solve_triangular(Rbb, R @ Z, upper=True, left=False)
            U, s, _ = torch.linalg.svd(Y, full_matrices=False)
            basis = U[:, :m]
        else:
            if case["sketch"] == "paper":
                S = torch.as_tensor(_normals(B.cpu().numpy(), k, i, 1, seed)[0], **dev)
                Om = torch.linalg.solve_triangular(LH[nI:, nI:].T, S, upper=True)
            else:
                t = torch.nonzero(plus)[:, 0]
                xi = torch.as_tensor(np.stack(_normals(t.cpu().numpy(), k, i, 0, seed),
                                              axis=1), **dev)
                f = torch.zeros((nn, k), **dev).index_add_(0, T[t].reshape(-1),
                                                           (Le[t] @ xi).reshape(-1, k))
                Om = torch.cholesky_solve(f[dofs], LH)[nI:]
            Y = R @ torch.cholesky_solve(A[:nI, nI:] @ Om, LA)[w]
            Qh, _ = torch.linalg.qr(Y)
            C = torch.zeros((nI, k), **dev)
            C[w] = R.T @ Qh
            t3 = A[nI:, :nI] @ torch.cholesky_solve(C, LA)
            Bm = torch.linalg.solve_triangular(LH[nI:, nI:], t3, upper=False)
            _, s, Uh = torch.linalg.svd(Bm, full_matrices=False)
            basis = Qh @ Uh.T[:, :m]
        cols = torch.linalg.solve_triangular(R, basis, upper=True)
        P = torch.nonzero(mine & free)[:, 0]
        pos = torch.searchsorted(W, P)
        Vi = torch.cat([u0[w][pos], cols[pos]], dim=1)
        lam, E = torch.linalg.eigh(Vi.T @ assemble(Ae, omega, P) @ Vi)
        good = lam > 1e-12 * lam[-1]
        kept.append(int(good.sum()))
        full = torch.zeros((nn, kept[-1]), **dev)
        full[P] = (Vi @ E[:, good]) / lam[good].sqrt()
        V.append(full)
        sig.append(s * s)
    V = torch.cat(V, dim=1)
    AV = torch.zeros_like(V)
    for t in torch.arange(nt, device="cuda").split(20000):
        AV.index_add_(0, T[t].reshape(-1), (Ae[t] @ V[T[t]]).reshape(4 * len(t), -1))
    K = V.T @ AV
    x = torch.linalg.solve(K, V.T @ load)
    wid = max(len(s) for s in sig) if case["explicit"] else widest
    sigma2 = torch.zeros((n_sub, wid), **dev)
    for i, s in enumerate(sig):
        sigma2[i, :len(s)] = s
    return (V @ x, sigma2.cpu().numpy(), np.asarray(kept, np.int32),
            float((V.T @ load) @ x))
