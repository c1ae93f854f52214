"""The work that this framework is measured on: products with the operator, solves and whole
scattering problems, through the calls that a user's program makes.

A case names the call ("call"), the problem (geometry, degree p, refinement level m, wavenumber
kappa, interpolation degree q), the form ("fp64": everything in double precision; "mixed": the
product in single precision) and the number of right-hand sides.  Results of the mixed form carry
single-precision digits in double-precision containers, and a program that chose it keeps them as
complex64; so that is what a mixed case returns.  The double-precision form returns complex128.

exact() is the same discrete problem written down plainly in 64 bits with torch: the quadrature
rules, the block tree and the interpolation of the operator's definition, without the library.
"""
import functools
import math

import numpy as np
import torch

from paper_1807_03097_gb300 import Solver
from paper_1807_03097_gb300.efie import Group, setup_many
from workloads import geometry as G

ETA = 1.6
# GMRES tolerance of the solves (relative), each form's to what its arithmetic can resolve: an iterate
# short of that depends on the order of rounding by much more than its digits are worth
TOL = {"fp64": 1e-12, "mixed": 1e-6}
FAR_DIRECTIONS = 64   # far-field directions of a whole scattering problem


def listed():
    return [
        # one product with the smallest operator in use (192 unknowns): launches and latency
        _case("matvec_small_fp64", "matvec", "sphere", 1, 2, 1.0, 4, "fp64"),
        # the default form (double precision) at an ordinary size
        _case("matvec_sphere_fp64", "matvec", "sphere", 2, 4, 10.0, 8, "fp64"),
        # the mixed form's product of every GMRES step of the 13k-unknown sphere
        _case("matvec_sphere_mixed", "matvec", "sphere", 2, 5, 10.0, 8, "mixed"),
        # higher wavenumber, degree and interpolation: 32 x 32 element blocks, 121 nodes
        _case("matvec_torus_mixed", "matvec", "torus", 3, 4, 20.0, 10, "mixed"),
        # the leaf-level option: most of the product is the near field
        _case("matvec_leafdense_mixed", "matvec", "sphere", 2, 4, 10.0, 8, "mixed", leaf_dense=1),
        # a few incident directions at once, a ragged count, a small tile
        _case("matvec_cube_r5_mixed", "matvec", "cube", 1, 4, 7.0, 6, "mixed", nrhs=5),
        # 64 incident directions at once
        _case("matvec_torus_r64_mixed", "matvec", "torus", 3, 3, 20.0, 10, "mixed", nrhs=64),
        # a new geometry or wavenumber: assembly, then the first product
        _case("assemble_sphere_fp64", "assemble", "sphere", 2, 4, 10.0, 8, "fp64"),
        # a solve in double precision with given right-hand side
        _case("solve_sphere_fp64", "solve", "sphere", 1, 3, 3.0, 5, "fp64"),
        # several directions solved in lockstep
        _case("solve_r6_mixed", "solve", "cube", 1, 3, 4.0, 6, "mixed", nrhs=6),
        # one request from geometry to far field
        _case("scatter_torus_mixed", "scatter", "torus", 1, 2, 3.0, 6, "mixed"),
        # independent problems of different size as one group
        _case("group_mixed", "group", "mix", 1, 3, 2.0, 6, "mixed", problems=8),
    ]


def _case(name, call, geometry, p, m, kappa, q, form, nrhs=1, leaf_dense=0, problems=0):
    return {"name": name, "call": call, "geometry": geometry, "p": p, "m": m, "kappa": kappa, "q": q, "form": form,
            "nrhs": nrhs, "leaf_dense": leaf_dense, "problems": problems}


def draw(rng):
    call = rng.choice(["matvec"] * 6 + ["assemble", "solve", "scatter", "group"])
    form = "mixed" if call == "group" else rng.choice(["mixed", "mixed", "fp64"])
    geometry = "mix" if call == "group" else rng.choice(["sphere", "cube", "torus"])
    nrhs = 1
    if call in ("matvec", "solve") and form == "mixed" and rng.random() < 0.4:
        nrhs = round(math.exp(rng.uniform(math.log(2), math.log(64 if call == "matvec" else 8))))
    while True:
        p, q = rng.choice([1, 1, 2, 2, 3]), rng.randint(3, 12 if form == "mixed" else 10)
        m = rng.randint(1, 5) if call in ("matvec", "assemble") else rng.randint(1, 3)
        if form == "mixed" and call in ("solve", "scatter", "group"):
            p = 1  # well conditioned: the iterates of the others differ by more than single precision
        elements = (16 if geometry == "torus" else 6) << (2 * m)
        tile = (q + 1) ** 4
        if call in ("solve", "scatter", "group"):
            if elements * tile <= (384 * 6 ** 4 if form == "fp64" else 384 * 7 ** 4) and p < 3:
                break
        elif elements * tile * max(1.0, nrhs / 8) <= 6144 * 9 ** 4 * (1.0 if form == "mixed" else 0.25) \
                and elements * (p + 1) ** 2 * (p + 4) ** 4 <= 6144 * 9 * 6 ** 4:
            break
    # solves stay below the scatterers' lowest interior resonances, where the system is singular
    low, high = (1.0, 20.0) if call in ("matvec", "assemble") else (0.8, 2.0)
    kappa = math.exp(rng.uniform(math.log(low), math.log(high)))
    dense = int(call == "matvec" and nrhs == 1 and elements <= 1536 and rng.random() < 0.2)
    c = _case("", call, geometry, p, m, kappa, q, form, nrhs, dense, rng.randint(2, 8) if call == "group" else 0)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------- the calls
def _patches(geometry, size):
    if geometry == "sphere":
        return G.sphere(size)
    return G.cube(2.0 * size) if geometry == "cube" else G.torus(2.0 * size, 0.5 * size)


def _problems(case, seed):
    """[(patches, options, directions, polarisations)]: what the seed decides.  Products and solves
    with a given operator keep the geometry and change the vectors; an assembly, a scattering
    problem and a group are of another size of scatterer and another incidence."""
    rng = np.random.default_rng(seed)
    fresh = case["call"] in ("assemble", "scatter", "group")
    out = []
    for k in range(max(1, case["problems"])):
        geometry, p, m, kappa = case["geometry"], case["p"], case["m"], case["kappa"]
        if geometry == "mix":  # a seeded order would change the work: the mix itself is fixed
            geometry, m = ("cube", "sphere", "torus")[k % 3], max(1, case["m"] - k // 3)
            m, kappa = m - (geometry == "torus" and m > 1), case["kappa"] * (0.4 + 0.6 * k / case["problems"])
        size = float(rng.uniform(0.98, 1.02)) if fresh else 1.0
        opts = dict(p=p, level_m=m, kappa=kappa, q=case["q"], eta=ETA, precision=int(case["form"] == "mixed"),
                    gmres_tol=TOL[case["form"]], leaf_dense=case["leaf_dense"])
        d, pol = G.plane_waves(case["nrhs"], int(rng.integers(1 << 30)))
        out.append((_patches(geometry, size), opts, d, pol))
    return out


def _directions(n):
    k = np.arange(n) + 0.5
    z, a = 1.0 - 2.0 * k / n, k * math.pi * (3.0 - math.sqrt(5.0))
    s = np.sqrt(1.0 - z * z)
    return np.stack([s * np.cos(a), s * np.sin(a), z], axis=1)


def _vectors(nrhs, n, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)
    x = torch.randn((nrhs, n, 2), dtype=torch.float64, device="cuda", generator=g)
    return torch.view_as_complex(x)


def prepare(case, seed):
    problems = _problems(case, seed)
    patches, opts, d, pol = problems[0]
    state = {"case": case, "d": d, "pol": pol}
    if case["call"] == "group":
        solvers = []
        for geo, o, _, _ in problems:
            solvers.append(Solver(None, **o))
            solvers[-1].set_geometry(geo)
        setup_many(solvers)
        state["group"] = Group(solvers)
        state["b"] = [torch.from_numpy(s.rhs(pr[2], pr[3])[0]).cuda() for s, pr in zip(solvers, problems)]
        return state
    if case["call"] in ("assemble", "scatter"):
        s = Solver(None, **opts)
        s.set_geometry(patches)
        if case["call"] == "assemble":
            n = 2 * len(patches) * ((1 << case["m"]) + case["p"] - 1) ** 2
            state["x"] = _vectors(1, n, seed)[0]
    else:
        s = Solver(patches, **opts)
        if case["call"] == "matvec":
            x = _vectors(case["nrhs"], s.ndof, seed)
            state["x"] = x if case["nrhs"] > 1 else x[0]
        else:
            b = torch.from_numpy(s.rhs(d, pol)).cuda()
            state["x"] = b if case["nrhs"] > 1 else b[0]
    state["solver"] = s
    return state


def run(state):
    case = state["case"]
    kept = (lambda v: v) if case["form"] == "fp64" else _single
    if case["call"] == "matvec":
        return kept(state["solver"].matvec(state["x"]))
    if case["call"] == "assemble":
        state["solver"].setup()
        return kept(state["solver"].matvec(state["x"]))
    if case["call"] == "solve":
        return kept(state["solver"].solve(state["x"])[0])
    if case["call"] == "scatter":
        s = state["solver"]
        s.setup()
        w = s.solve_plane_waves(state["d"], state["pol"])[0]
        return [kept(w), kept(s.far_field(w, _directions(FAR_DIRECTIONS)))]
    return [kept(x) for x in state["group"].solve(state["b"])[0]]


def _single(v):
    return v.to(torch.complex64) if isinstance(v, torch.Tensor) else v.astype(np.complex64)


# ---------------------------------------------------------------------------------------- the work
PRODUCTS = 100  # products of one solve (GMRES steps), about


def work(case):
    """Per product: every admissible block's kernel entries applied to 4 complex fields (8 flop each,
    and 16 to evaluate an entry where none is kept), every near block once.  Per assembly: the
    quadrature points' kernel and geometry (200 flop a point) and the blocks written."""
    total = {"bytes": 0.0, "flops": 0.0}
    for patches, o, _, _ in _problems(case, 0):
        size = 16 if o["precision"] == 0 else 8
        far, near, points = _counts(_key(case, o, len(patches)), case["leaf_dense"])
        p1, nodes = o["p"] + 1, (o["q"] + 1) ** 2
        nb, n = 2 * p1 * p1, 2 * len(patches) * ((1 << o["level_m"]) + o["p"] - 1) ** 2
        r, products = case["nrhs"], 1 if case["call"] in ("matvec", "assemble") else PRODUCTS
        total["flops"] += products * (far * nodes ** 2 * (32.0 * r + (16 if size == 8 else 0)) + near * nb * nb * 8.0 * r)
        total["bytes"] += products * (near * nb * nb * size + 32.0 * n * r)
        if case["call"] in ("assemble", "scatter"):
            total["flops"] += 200.0 * points
            total["bytes"] += near * nb * nb * 16.0
    return total


def _key(case, o, n_patches):
    return ({6: "cube", 16: "torus"}[n_patches] if case["geometry"] == "mix" else case["geometry"], o["p"], o["level_m"], o["q"])


@functools.lru_cache(maxsize=None)
def _counts(key, leaf_dense):
    geometry, p, m, q = key
    e = _Exact(_patches(geometry, 1.0), p, m, 1.0, q, leaf_dense, "cpu", tree_only=True)
    kinds = e.kind[e.near[:, 0] <= e.near[:, 1]]
    g4 = (p + 4) ** 4
    return len(e.far), len(e.near), float(sum(int((kinds == k).sum()) * n * g4 for k, n in ((0, 1), (1, 4), (2, 6), (3, 8))))


# ---------------------------------------------------------------------------------------- in 64 bits
def exact(case, seed):
    out = []
    for k, (patches, o, d, pol) in enumerate(_problems(case, seed)):
        e = _Exact(patches, o["p"], o["level_m"], o["kappa"], o["q"], o["leaf_dense"], "cuda" if torch.cuda.is_available() else "cpu")
        if case["call"] in ("matvec", "assemble"):
            x = _vectors(case["nrhs"], e.ndof, seed)
            y = e.product(x)
            return y if case["nrhs"] > 1 else y[0]
        x = torch.linalg.solve(e.matrix(), e.plane_waves(d, pol).T.contiguous()).T.contiguous()
        if case["call"] == "solve":
            return x if case["nrhs"] > 1 else x[0]
        if case["call"] == "scatter":
            return [x, e.far_field(x, _directions(FAR_DIRECTIONS))]
        out.append(x[0])
    return out


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _bernstein(p, t):
    """Values and derivatives [..., p + 1] of the Bernstein polynomials of degree p."""
    def values(d):
        return torch.stack([math.comb(d, a) * t ** a * (1 - t) ** (d - a) for a in range(d + 1)], -1)
    if p == 0:
        return torch.ones_like(t)[..., None], torch.zeros_like(t)[..., None]
    low, zero = values(p - 1), torch.zeros_like(t)[..., None]
    return values(p), p * (torch.cat([zero, low], -1) - torch.cat([low, zero], -1))


def _lagrange(nodes, t):
    """[len(t), len(nodes)] values of the Lagrange polynomials of `nodes` at `t`."""
    return np.stack([np.prod([(t - nodes[k]) / (nodes[i] - nodes[k]) for k in range(len(nodes)) if k != i], axis=0)
                     for i in range(len(nodes))], axis=1)


def _spread(k):
    """The two coordinates of a place in the quadtree order (bits in turn, first coordinate lowest)."""
    a, b = k * 0, k * 0
    for t in range(12):
        a, b = a | (((k >> (2 * t)) & 1) << t), b | (((k >> (2 * t + 1)) & 1) << t)
    return a, b


def _duffy(kind, x, w):
    """Points (s, t) in two unit squares [n, 2] and weights [n] for pairs of elements that lie apart
    (0), share a vertex at the origin (1), share the edge {s2 = 0} = {t2 = 0} (2) or coincide (3)."""
    a, b, c, d = (v.reshape(-1) for v in np.meshgrid(x, x, x, x, indexing="ij"))
    w4 = functools.reduce(np.multiply, (v.reshape(-1) for v in np.meshgrid(w, w, w, w, indexing="ij")))
    parts = []
    if kind == 0:
        parts.append((a, b, c, d, w4))
    if kind == 1:
        for big in range(4):
            v = [a * b, a * c, a * d]
            v.insert(big, a)
            parts.append((*v, w4 * a ** 3))
    if kind == 2:
        for sign in (1, -1):
            for z, s2, t2 in ((a, a * b, a * c), (a * b, a, a * c), (a * b, a * c, a)):
                s1 = (z if sign < 0 else 0.0) + (1 - z) * d
                parts.append((s1, s2, s1 + sign * z, t2, w4 * a * a * (1 - z)))
    if kind == 3:
        for i in range(8):
            z0, z1 = (a, a * b) if i < 4 else (a * b, a)
            g0, g1 = (-1 if i & 1 else 1), (-1 if i & 2 else 1)
            s1, s2 = (z0 if g0 < 0 else 0.0) + (1 - z0) * c, (z1 if g1 < 0 else 0.0) + (1 - z1) * d
            parts.append((s1, s2, s1 + g0 * z0, s2 + g1 * z1, w4 * a * (1 - z0) * (1 - z1)))
    s1, s2, t1, t2, wt = (np.concatenate([q[i] for q in parts]) for i in range(5))
    return np.stack([s1, s2], 1), np.stack([t1, t2], 1), wt


def _turn(code, s):
    """The square's symmetry `code` [N] (swap, then reflections) applied to points s [n, 2] -> [N, n, 2]."""
    a = torch.where((code & 1).bool()[:, None], s[None, :, 1], s[None, :, 0])
    b = torch.where((code & 1).bool()[:, None], s[None, :, 0], s[None, :, 1])
    a = torch.where((code & 2).bool()[:, None], 1 - a, a)
    return torch.stack([a, torch.where((code & 4).bool()[:, None], 1 - b, b)], -1)


class _Exact:
    """The discrete operator of one problem in double precision: superspace blocks of the near pairs
    by quadrature, admissible blocks by tensor Chebyshev interpolation, glued by T."""

    def __init__(self, patches, p, m, kappa, q, leaf_dense, device, tree_only=False):
        self.p, self.m, self.n, self.kappa, self.q1 = p, m, 1 << m, kappa, q + 1
        self.np, self.p1, self.g, self.device = len(patches), p + 1, p + 4, device
        self.nE, self.nb, self.nI = self.np * self.n ** 2, 2 * (p + 1) ** 2, (q + 1) ** 2
        # all patches are Bezier patches of one bidegree: homogeneous control nets [patch][b][a][4]
        self.deg = patches[0]["deg"]
        self.net = self._t(np.stack([np.concatenate([pt["cp"] * pt["w"][..., None], pt["w"][..., None]], -1) for pt in patches]))
        self._tree(leaf_dense)
        self._touching()
        if tree_only:
            return
        self._glue()
        self._blocks()
        self._tables()

    def _t(self, a):
        return torch.as_tensor(a, device=self.device)

    def at(self, patch, s):
        """F and its two derivatives at s [..., 2] of patch [...]: [..., 3], [..., 2, 3]."""
        u, du = _bernstein(self.deg[0], s[..., 0])
        v, dv = _bernstein(self.deg[1], s[..., 1])
        net = self.net[patch]
        r, ru = torch.einsum("...bak,...a->...bk", net, u), torch.einsum("...bak,...a->...bk", net, du)
        f, f1, f2 = (torch.einsum("...bk,...b->...k", x, y) for x, y in ((r, v), (ru, v), (r, dv)))
        x = f[..., :3] / f[..., 3:]
        return x, torch.stack([(f1[..., :3] - x * f1[..., 3:]) / f[..., 3:], (f2[..., :3] - x * f2[..., 3:]) / f[..., 3:]], -2)

    def _place(self, level):
        """Patch and lower corner, in cells, of every cluster of a level."""
        k = torch.arange(self.np << (2 * level), device=self.device)
        i, j = _spread(k & ((1 << (2 * level)) - 1))
        return k >> (2 * level), torch.stack([i, j], -1).to(torch.float64)

    def _tree(self, leaf_dense):
        grid = torch.linspace(0, 1, 9, dtype=torch.float64, device=self.device)
        grid = torch.cartesian_prod(grid, grid)
        balls = []
        for l in range(self.m + 1):
            patch, low = self._place(l)
            c = self.at(patch, (low + 0.5) / (1 << l))[0]
            r = torch.stack([(self.at(patch, (low + g) / (1 << l))[0] - c).norm(dim=-1) for g in grid]).amax(0)
            balls.append((c, r))
        dense = leaf_dense and self.p1 ** 2 < self.nI
        k = torch.arange(self.np, device=self.device)
        pair, far, self.level_far = torch.cartesian_prod(k, k), [], []
        for l in range(self.m + 1):
            c, r = balls[l]
            d = (c[pair[:, 0]] - c[pair[:, 1]]).norm(dim=-1) - r[pair[:, 0]] - r[pair[:, 1]]
            ok = (d > 0) & (2 * torch.maximum(r[pair[:, 0]], r[pair[:, 1]]) <= ETA * d)
            if dense and l == self.m:
                ok = torch.zeros_like(ok)
            self.level_far.append(pair[ok])
            pair = pair[~ok]
            if l < self.m:
                four = torch.arange(4, device=self.device)
                ch = torch.cartesian_prod(four, four)
                pair = (4 * pair[:, None, :] + ch[None]).reshape(-1, 2)
        self.near, self.far = pair, torch.cat(self.level_far)

    def _touching(self):
        """Kind and symmetry codes of every near pair."""
        patch, low = self._place(self.m)
        corner = torch.stack([self.at(patch, (low + self._t(np.array(v))) / self.n)[0]
                              for v in ((0, 0), (1, 0), (0, 1), (1, 1))], 1)      # [element][corner][3]
        tol = 1e-9 * float((corner.reshape(-1, 3).amax(0) - corner.reshape(-1, 3).amin(0)).norm())
        e, f = self.near[:, 0], self.near[:, 1]
        same = (corner[e][:, :, None] - corner[f][:, None, :]).norm(dim=-1) < tol
        count = same.reshape(-1, 16).sum(1)
        self.kind = torch.where(e == f, 3, count)
        self.code = torch.zeros_like(self.near)
        maps = {}  # (corner that the origin goes to, corner that (1, 0) goes to) -> code
        for code in range(8):
            def go(u, v, code=code):
                a, b = (v, u) if code & 1 else (u, v)
                return (1 - a if code & 2 else a) + 2 * (1 - b if code & 4 else b)
            maps[go(0, 0), go(1, 0)] = code
        one = self.kind == 1
        first = same[one].reshape(-1, 16).to(torch.int64).argmax(1)
        for side, at in ((0, first // 4), (1, first % 4)):
            self.code[one, side] = ((at & 1) << 1) | ((at >> 1) << 2)
        two = torch.nonzero(self.kind == 2).reshape(-1)
        hits = same[two].reshape(-1, 16).nonzero()[:, 1].reshape(-1, 2)
        a, b = hits // 4, hits % 4                                                # the two common corners
        pa = corner[e[two]][torch.arange(len(two), device=self.device)[:, None], a]
        diff = pa[:, 1] - pa[:, 0]
        big = diff.abs() > tol
        lead = torch.gather(diff, 1, big.to(torch.int64).argmax(1, keepdim=True))[:, 0]
        swap = (lead < 0)[:, None]
        a, b = torch.where(swap, a.flip(1), a), torch.where(swap, b.flip(1), b)
        table = torch.zeros(16, dtype=torch.int64)
        for (u, v), code in maps.items():
            table[4 * u + v] = code
        table = table.to(self.device)
        self.code[two, 0], self.code[two, 1] = table[4 * a[:, 0] + a[:, 1]], table[4 * b[:, 0] + b[:, 1]]

    def _basis(self, s):
        """psi [..., NS] and its two derivatives [..., 2, NS] at element coordinates s."""
        u, du = _bernstein(self.p, s[..., 0])
        v, dv = _bernstein(self.p, s[..., 1])
        flat = lambda x, y: (y[..., :, None] * x[..., None, :]).flatten(-2)  # noqa: E731
        return flat(u, v), torch.stack([flat(du, v), flat(u, dv)], -2)

    def _sides(self, element, s):
        """T[pair, point, k, (alpha, ab)] = h^2 d_alpha F_k psi (k < 3), h d_alpha psi (k = 3); and F."""
        h = 1.0 / self.n
        patch, low = self._place(self.m)
        x, d = self.at(patch[element][:, None].expand(s.shape[:-1]), (low[element][:, None, :] + s) * h)
        psi, dpsi = self._basis(s)
        geo = h * h * d.transpose(-1, -2)[..., None] * psi[..., None, None, :]      # [..., 3, 2, NS]
        return torch.cat([geo, h * dpsi[..., None, :, :]], -3).flatten(-2), x

    def _blocks(self):
        """Near blocks [pair, row, column], complex; those with e > e' are the transposes."""
        x, w = _gauss(self.g)
        self.block = torch.zeros((len(self.near), self.nb, self.nb), dtype=torch.complex128, device=self.device)
        key = self.near[:, 0] * self.nE + self.near[:, 1]
        order = key.argsort()
        twin = order[torch.searchsorted(key[order], self.near[:, 1] * self.nE + self.near[:, 0])]
        sign = self._t(np.array([1.0, 1.0, 1.0, -1.0 / self.kappa ** 2]))
        upper = self.near[:, 0] <= self.near[:, 1]
        for kind in range(4):
            s, t, wt = (self._t(v) for v in _duffy(kind, x, w))
            todo = torch.nonzero(upper & (self.kind == kind)).reshape(-1)
            for part in todo.split(max(1, 2_000_000 // (len(wt) * self.nb))):
                e, f = self.near[part, 0], self.near[part, 1]
                ts, xs = self._sides(e, _turn(self.code[part, 0], s))
                tt, xt = self._sides(f, _turn(self.code[part, 1], t))
                r = (xs - xt).norm(dim=-1)
                g = wt / (4 * math.pi * r)
                right = (tt * sign[:, None]).flatten(1, 2)
                left = [(ts * (g * fn(self.kappa * r))[..., None, None]).flatten(1, 2).transpose(1, 2) for fn in (torch.cos, torch.sin)]
                self.block[part] = torch.complex(left[0] @ right, left[1] @ right)
        self.block[~upper] = self.block[twin[~upper]].transpose(1, 2)

    def _tables(self):
        q1, p1 = self.q1, self.p1
        nodes = 0.5 - 0.5 * np.cos(math.pi * (2 * np.arange(q1) + 1) / (2.0 * q1))
        x, w = _gauss(q1 + p1 + 1)
        b, db = _bernstein(self.p, torch.from_numpy(x))
        lag = _lagrange(nodes, x)
        c = torch.complex128
        self.M, self.Md = self._t(lag.T @ (w[:, None] * b.numpy())).to(c), self._t(lag.T @ (w[:, None] * db.numpy())).to(c)
        self.E = self._t(np.stack([_lagrange(nodes, 0.5 * (ch + nodes)).T for ch in (0, 1)])).to(c)  # [child][m][m']
        tensor = self._t(np.stack([np.tile(nodes, q1), np.repeat(nodes, q1)], 1))
        self.node = []
        for l in range(self.m + 1):
            patch, low = self._place(l)
            self.node.append(self.at(patch[:, None].expand(-1, self.nI), (low[:, None, :] + tensor) / (1 << l)))

    def superspace(self, xs):
        """(N + F) xs for xs [R, nE, 2, p1, p1]."""
        R, q1, h, c = xs.shape[0], self.q1, 1.0 / self.n, torch.complex128
        ys = torch.zeros((self.nE, self.nb, R), dtype=c, device=self.device)
        flat = xs.reshape(R, self.nE, self.nb).permute(1, 2, 0).contiguous()
        for part in torch.arange(len(self.near), device=self.device).split(max(1, (1 << 28) // (self.nb * (R + self.nb)))):
            ys.index_add_(0, self.near[part, 0], self.block[part] @ flat[self.near[part, 1]])
        ys = ys.permute(2, 0, 1).reshape(xs.shape)
        two = lambda a, b, v: torch.einsum("nb,ma,reba->renm", a, b, v)  # noqa: E731
        M, Md = self.M, self.Md
        mom = torch.stack([h * h * two(M, M, xs[:, :, 0]), h * h * two(M, M, xs[:, :, 1]),
                           h * (two(M, Md, xs[:, :, 0]) + two(Md, M, xs[:, :, 1]))], 2)          # [R, e, 3, m2, m1]
        moms = [mom]
        for l in range(self.m, 0, -1):
            ch = moms[-1].reshape(R, -1, 4, 3, q1, q1)
            moms.append(sum(torch.einsum("nj,mi,refji->refnm", self.E[k >> 1], self.E[k & 1], ch[:, :, k]) for k in range(4)))
        moms.reverse()
        loc = None
        for l in range(self.m + 1):
            x, d = self.node[l]
            mu = moms[l].flatten(-2)                                                             # [R, e, 3, nI]
            src = torch.cat([torch.einsum("emak,ream->remk", d.to(c), mu[:, :, :2]), mu[:, :, 2, :, None]], -1)
            src = src.permute(1, 2, 0, 3).reshape(len(x), self.nI, 4 * R)
            acc = torch.zeros_like(src)
            pairs = self.level_far[l]
            for part in pairs.split(max(1, (1 << 27) // (self.nI * (self.nI + 8 * R)))):
                r = (x[part[:, 0]][:, :, None] - x[part[:, 1]][:, None, :]).norm(dim=-1)
                acc.index_add_(0, part[:, 0], torch.polar(0.25 / (math.pi * r), self.kappa * r) @ src[part[:, 1]])
            acc = acc.reshape(len(x), self.nI, R, 4).permute(2, 0, 1, 3)
            new = torch.cat([torch.einsum("emak,remk->ream", d.to(c), acc[..., :3]), -acc[..., 3][:, :, None] / self.kappa ** 2], 2)
            new = new.reshape(R, len(x), 3, q1, q1)
            if loc is not None:
                new += torch.stack([torch.einsum("nj,mi,refnm->refji", self.E[k >> 1], self.E[k & 1], loc) for k in range(4)], 2).flatten(1, 2)
            loc = new
        back = lambda a, b, v: torch.einsum("nb,ma,renm->reba", a, b, v)  # noqa: E731
        ys = ys + torch.stack([h * h * back(M, M, loc[:, :, 0]) + h * back(M, Md, loc[:, :, 2]),
                               h * h * back(M, M, loc[:, :, 1]) + h * back(Md, M, loc[:, :, 2])], 2)
        return ys

    def _glue(self):
        """T as a sparse real matrix: Bernstein coefficients of the div-conforming splines, those on a
        common edge of two patches glued with the sign that keeps the normal flux continuous."""
        n, p, p1 = self.n, self.p, self.p1
        t = np.linspace(0, 1, 5)
        one = np.ones(5)
        line = [np.stack(v, 1) for v in ((0 * one, t), (one, t), (t, 0 * one), (t, one))]
        pts = np.stack([[self.at(torch.full((5,), j, device=self.device), self._t(v))[0].cpu().numpy() for v in line] for j in range(self.np)])
        pts = pts.reshape(4 * self.np, 5, 3)
        tol = 1e-7 * np.linalg.norm(pts.reshape(-1, 3).max(0) - pts.reshape(-1, 3).min(0))
        other = {}
        for a in range(4 * self.np):
            for b in range(4 * self.np):
                for rev in (0, 1):
                    if a != b and np.abs(pts[a] - (pts[b][::-1] if rev else pts[b])).max() < tol:
                        other[a] = (b, rev)
        shape = [(n + p - 1, n + p), (n + p, n + p - 1)]                         # [i2][i1] of the two components
        count = (n + p) * (n + p - 1)
        flat = lambda j, comp, i1, i2: (2 * j + comp) * count + i2 * shape[comp][1] + i1  # noqa: E731
        edge = lambda j, k, pos: flat(j, k // 2, *((0 if k == 0 else n + p - 1, pos) if k < 2 else (pos, 0 if k == 2 else n + p - 1)))  # noqa: E731
        twin = np.full(2 * count * self.np, -1)
        sign = np.ones(2 * count * self.np)
        for a, (b, rev) in other.items():
            for pos in range(n + p - 1):
                i, j = edge(a // 4, a % 4, pos), edge(b // 4, b % 4, n + p - 2 - pos if rev else pos)
                if j < i:
                    twin[i] = j
                    sign[i] = -(1 if a % 4 in (1, 3) else -1) * (1 if b % 4 in (1, 3) else -1)
        dof = np.cumsum(twin < 0) - 1
        dof = np.where(twin < 0, dof, dof[twin])
        self.ndof = int((twin < 0).sum())

        def extraction(degree):
            """[element][a][r]: coefficient of B_a in the spline k + r of open equidistant knots."""
            kn = np.clip((np.arange(n + 2 * degree + 1) - degree) / n, 0, 1)
            x, _ = _gauss(p1)
            inv = np.linalg.inv(_bernstein(p, torch.from_numpy(x))[0].numpy())
            out = np.zeros((n, p1, degree + 1))
            for k in range(n):
                y = (k + x) / n
                val = [((i == k + degree) * np.ones(p1)) for i in range(n + 2 * degree)]
                for d in range(1, degree + 1):
                    val = [sum(((y - kn[i]) / (kn[i + d] - kn[i]) * val[i] if kn[i + d] > kn[i] else 0.0,
                                (kn[i + d + 1] - y) / (kn[i + d + 1] - kn[i + 1]) * val[i + 1] if kn[i + d + 1] > kn[i + 1] else 0.0))
                           for i in range(len(val) - 1)]
                for r in range(degree + 1):
                    out[k, :, r] = inv @ (val[k + r] * np.ones(p1))
            return out
        up, lo = extraction(p), extraction(p - 1)
        rows, cols, vals = [], [], []
        i1, i2 = _spread(np.arange(n * n))
        for comp in (0, 1):
            c1, c2 = (up, lo) if comp == 0 else (lo, up)
            v = c2[i2][:, :, None, :, None] * c1[i1][:, None, :, None, :]         # [e][b][a][r2][r1]
            e, b, a, r2, r1 = np.indices(v.shape)
            for j in range(self.np):
                f = flat(j, comp, i1[e] + r1, i2[e] + r2)
                rows.append(((((j * n * n + e) * 2 + comp) * p1 + b) * p1 + a).reshape(-1))
                cols.append(dof[f].reshape(-1))
                vals.append((v * sign[f]).reshape(-1))
        rows, cols, vals = (np.concatenate(v) for v in (rows, cols, vals))
        self.T = torch.sparse_coo_tensor(self._t(np.stack([rows, cols])), self._t(vals).to(torch.complex128), (self.nE * self.nb, self.ndof), check_invariants=False).coalesce()
        self.Tt = self.T.transpose(0, 1).coalesce()

    def _down(self, x):
        return (self.T @ x.T).T.reshape(-1, self.nE, 2, self.p1, self.p1).contiguous()

    def _up(self, ys):
        return (self.Tt @ ys.reshape(len(ys), -1).T).T.contiguous()

    def product(self, x):
        return self._up(self.superspace(self._down(x)))

    def matrix(self):
        eye = torch.eye(self.ndof, dtype=torch.complex128, device=self.device)
        return torch.cat([self.product(part) for part in eye.split(256)]).T.contiguous()

    def _points(self):
        """Gauss points of every element: F [e, g, 3], derivatives, weights h^2 w [g], psi [g, NS]."""
        x, w = _gauss(self.g)
        s = self._t(np.stack([np.tile(x, self.g), np.repeat(x, self.g)], 1))
        patch, low = self._place(self.m)
        f, d = self.at(patch[:, None].expand(-1, len(s)), (low[:, None, :] + s) / self.n)
        return f, d, self._t(np.outer(w, w).reshape(-1)) / self.n ** 2, self._basis(s)[0]

    def plane_waves(self, dirs, pols):
        f, d, w, psi = self._points()
        out = []
        for k, pol in zip(self._t(np.asarray(dirs)), self._t(np.asarray(pols))):
            wave = torch.polar(torch.ones_like(f[..., 0]), self.kappa * (f @ k))
            out.append(-torch.einsum("eg,ega,g,gn->ean", wave, (d @ pol).to(wave.dtype), w.to(wave.dtype), psi.to(wave.dtype)))
        return self._up(torch.stack(out))

    def far_field(self, x, dirs):
        f, d, w, psi = self._points()
        c = torch.complex128
        amp = self._down(x).reshape(len(x), self.nE, 2, -1)
        cur = torch.einsum("rean,gn,egak,g->regk", amp, psi.to(c), d.to(c), w.to(c))
        out = []
        for k in self._t(np.asarray(dirs)):
            W = torch.einsum("eg,regk->rk", torch.polar(torch.ones_like(f[..., 0]), -self.kappa * (f @ k)), cur)
            out.append((W - k * (W @ k.to(c))[:, None]) / (4 * math.pi))
        return torch.stack(out, 1)
