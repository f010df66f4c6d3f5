"""The work that users of the node-patch Poisson-Boltzmann library have it do.

A case names a molecule (a geodesic sphere, a globular molecule's isosurface, or a cluster
of globules), the library's options and one use of it:

* product -- y = L x through ``Handle.matvec`` on device buffers: what every GMRES iteration
             costs, and the product a caller with an iteration of their own calls;
* host    -- the same product through ``Handle.matvec_host`` from and to pinned host memory;
* solve   -- ``Handle.solve`` and ``Handle.energy`` on a handle that exists;
* request -- one molecule from its mesh to its energy: handle, solve, energy;
* batch   -- ``solve_batch`` over several molecules at once.

The seed turns the molecule (a rigid rotation, so that each seed has another octree) and
draws the unknowns.
"""
import functools
import math

import numpy as np
import torch

import paper_1710_06316_gb300 as pb

KAPPA = 0.104            # 1/Angstrom, 100 mM salt
NEAR_C = 2.0             # the library's default near-set factor
COULOMB = 332.0636       # kcal Angstrom / (mol e^2)
EXACT_NODES = 210000     # the FP64 sums take all pairs of nodes
EXACT_DENSE = 36000      # FP64 solves keep the dense operator


# ---- cases --------------------------------------------------------------------------------
def listed():
    return [
        # the smallest product: a single ion's sphere, where launches and latency count
        dict(name="product ion 2562", use="product", shape="sphere", freq=16, radius=2.0, atoms=1, eps_in=1.0,
             kappa=KAPPA, order=6, precision=1),
        # a peptide-sized isosurface (odd leaf sizes, lists 3 and 4 in use)
        dict(name="product peptide 12k", use="product", shape="globule", atoms=40, grid=0.4, eps_in=2.0,
             kappa=KAPPA, order=6, precision=1),
        # the workload that the library's product throughput is quoted on
        dict(name="product sphere 164k", use="product", shape="sphere", freq=128, radius=20.0, atoms=64, eps_in=2.0,
             kappa=KAPPA, order=6, precision=1),
        # the same in plain FP32, for callers who keep the tensor cores out of it
        dict(name="product sphere 164k fp32", use="product", shape="sphere", freq=128, radius=20.0, atoms=64,
             eps_in=2.0, kappa=KAPPA, order=6, precision=0),
        # a protein's isosurface
        dict(name="product protein 200k", use="product", shape="globule", atoms=1600, grid=0.4, eps_in=2.0,
             kappa=KAPPA, order=6, precision=1),
        # the accurate end of the order sweep, on a small protein
        dict(name="product protein 33k order 8", use="product", shape="globule", atoms=170, grid=0.4, eps_in=2.0,
             kappa=KAPPA, order=8, precision=1),
        # no salt (kappa = 0), a large single sphere
        dict(name="product sphere 655k no salt", use="product", shape="sphere", freq=256, radius=50.0, atoms=1,
             eps_in=2.0, kappa=0.0, order=6, precision=1),
        # a virus-capsid-like assembly: 60 separate closed surfaces
        dict(name="product assembly 5M", use="product", shape="cluster", copies=60, atoms=5500, grid=1.0, eps_in=2.0,
             kappa=KAPPA, order=6, precision=1),
        # a caller whose vectors live on the host
        dict(name="host product sphere 41k", use="host", shape="sphere", freq=64, radius=20.0, atoms=64, eps_in=2.0,
             kappa=KAPPA, order=6, precision=1),
        # one GMRES solve and the solvation energy of a small protein on an existing handle
        dict(name="solve protein 33k", use="solve", shape="globule", atoms=170, grid=0.4, eps_in=2.0, kappa=KAPPA,
             order=6, precision=1),
        # a serving request: a new molecule from its mesh to its energy
        dict(name="request protein 20k", use="request", shape="globule", atoms=1100, grid=1.0, eps_in=2.0,
             kappa=0.15, order=6, precision=1),
        # several small molecules solved together
        dict(name="batch 8 x 12k", use="batch", shape="globule", count=8, atoms=40, grid=0.4, eps_in=2.0, kappa=KAPPA,
             order=6, precision=1),
    ]


def draw(rng):
    """One more case of the ranges above."""
    use = rng.choice(["product"] * 6 + ["host", "solve", "request", "batch"])
    case = dict(use=use, eps_in=rng.choice([1.0, 2.0, 4.0]), kappa=rng.choice([0.03, KAPPA, 0.3]), order=6,
                precision=rng.choice([1, 1, 1, 0]))
    if use in ("product", "host"):
        case.update(order=rng.choice([4, 6, 6, 6, 8]), kappa=rng.choice([0.0, 0.03, KAPPA, 0.3]))
    top = {"product": 1e6, "host": 3e5, "solve": 6e4, "request": 6e4, "batch": 2e4}[use]   # nodes
    low = 600 if use in ("product", "host") else 2600
    nodes = low * (top / low) ** rng.random()
    if use == "batch":
        case["count"] = rng.randrange(2, 9)
    if rng.random() < 0.5:
        freq = round(math.sqrt(nodes / 10))
        case.update(shape="sphere", freq=freq, radius=round(rng.uniform(1.5, 3.0) * (freq / 16) ** 0.8, 3),
                    atoms=rng.randrange(20, 100))
    else:
        grid = rng.choice([0.4, 0.5, 0.7, 1.0])
        case.update(shape="globule", grid=grid, atoms=max(20, round((nodes * (grid / 0.4) ** 2 / 500) ** (1 / 0.81))))
    return case


# ---- molecules ----------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _sphere(freq):
    """Geodesic icosahedron on the unit sphere: 10 freq^2 + 2 nodes, 20 freq^2 triangles."""
    g = (1 + math.sqrt(5)) / 2
    corner = np.array([(s, t * g, 0.0) for s in (-1, 1) for t in (-1, 1)])
    corner = np.concatenate([np.roll(corner, k, axis=1) for k in range(3)])
    edge = np.abs(np.linalg.norm(corner[:, None] - corner[None], axis=2) - 2.0) < 1e-6
    faces = [(i, j, k) for i in range(12) for j in range(i) for k in range(j) if edge[i, j] and edge[j, k] and edge[i, k]]
    spots = [(i, j) for i in range(freq + 1) for j in range(freq + 1 - i)]
    at = np.zeros((freq + 1, freq + 1), np.int64)
    at[tuple(np.array(spots).T)] = np.arange(len(spots))
    weights = np.array([(freq - i - j, i, j) for i, j in spots], float) / freq
    small = [(at[i, j], at[i + 1, j], at[i, j + 1]) for i in range(freq) for j in range(freq - i)]
    small += [(at[i + 1, j], at[i + 1, j + 1], at[i, j + 1]) for i in range(freq - 1) for j in range(freq - 1 - i)]
    small = np.array(small)
    points, tri = [], []
    for n, (i, j, k) in enumerate(faces):
        a, b, c = corner[i], corner[j], corner[k]
        if np.dot(np.cross(b - a, c - a), a) < 0:
            b, c = c, b
        points.append(weights @ np.stack([a, b, c]))
        tri.append(small + n * len(spots))
    points, tri = np.concatenate(points), np.concatenate(tri)
    cell = np.floor(points * 2.0 ** 17 + 0.1371).astype(np.int64) + (1 << 19)   # faces share their edges' nodes
    _, first, back = np.unique((cell[:, 0] << 40) + (cell[:, 1] << 20) + cell[:, 2], return_index=True, return_inverse=True)
    xyz = points[first]
    return xyz / np.linalg.norm(xyz, axis=1, keepdims=True), back.reshape(-1)[tri].astype(np.int32)


def _isosurface(value, origin, step):
    """The surface value = 0 on a regular grid (inside: value > 0), by six tetrahedra to a cube."""
    shape = np.array(value.shape)
    flat, stride = value.reshape(-1), np.array([shape[1] * shape[2], shape[2], 1])
    inside = value > 0
    count = sum(inside[a:shape[0] - 1 + a, b:shape[1] - 1 + b, c:shape[2] - 1 + c].astype(np.int8)
                for a in (0, 1) for b in (0, 1) for c in (0, 1))
    cube = np.stack(np.nonzero((count > 0) & (count < 8)), 1) @ stride
    tets = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):   # paths from corner 0 to corner 7
        tets.append(np.stack([cube + stride[list(p[:k])].sum() for k in range(4)], 1).astype(np.int64))
    tets = np.concatenate(tets)
    tets = np.take_along_axis(tets, np.argsort(flat[tets] <= 0, axis=1, kind="stable"), 1)   # inside corners first
    number = (flat[tets] > 0).sum(1)

    def place(p):
        return origin + step * np.stack([p // stride[0], p // stride[1] % shape[1], p % shape[2]], -1)

    ends = []
    for n, cuts in ((1, [(0, 1, 0, 2, 0, 3)]), (2, [(0, 2, 0, 3, 1, 3), (0, 2, 1, 3, 1, 2)]), (3, [(0, 3, 1, 3, 2, 3)])):
        part = tets[number == n]
        if len(part):
            out = place(part[:, n:]).mean(1) - place(part[:, :n]).mean(1)
            for cut in cuts:
                ends.append((part[:, list(cut)].reshape(-1, 3, 2), out))
    out = np.concatenate([o for _, o in ends])
    ends = np.concatenate([e for e, _ in ends])                 # [triangle, corner, (inside end, outside end)]
    size = np.int64(flat.size)
    _, first, back = np.unique((ends[..., 0] * size + ends[..., 1]).reshape(-1), return_index=True, return_inverse=True)
    a, b = ends.reshape(-1, 2)[first].T
    t = np.clip(flat[a] / (flat[a] - flat[b]), 0.2, 0.8)[:, None]   # no slivers
    xyz = place(a) * (1 - t) + place(b) * t
    tri = back.reshape(-1, 3)
    p = xyz[tri]
    flip = (np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]) * out).sum(1) < 0
    tri[flip] = tri[flip][:, [0, 2, 1]]
    return xyz, tri


def _outer_and_smooth(xyz, tri):
    """The connected surface with the largest x, after ten of Taubin's smoothing passes (0.5, -0.53)."""
    n = len(xyz)
    u = np.concatenate([tri[:, [0, 1]], tri[:, [1, 2]], tri[:, [2, 0]]])
    u, v = torch.from_numpy(u[:, 0].copy()), torch.from_numpy(u[:, 1].copy())   # each edge once in each direction
    label = torch.arange(n)
    while True:
        least = torch.minimum(label[u], label[v])
        new = label.scatter_reduce(0, u, least, "amin").scatter_reduce(0, v, least, "amin")
        new = new.scatter_reduce(0, label, new, "amin")[label]   # the whole of an old part moves
        if torch.equal(new, label):
            break
        label = new
    label = label.numpy()
    tri = tri[label[tri[:, 0]] == label[np.argmax(xyz[:, 0])]]
    used, tri = np.unique(tri, return_inverse=True)
    xyz, tri = xyz[used], tri.reshape(-1, 3)
    u = np.concatenate([tri[:, 0], tri[:, 1], tri[:, 2]])
    v = np.concatenate([tri[:, 1], tri[:, 2], tri[:, 0]])
    degree = np.bincount(u, minlength=len(xyz))[:, None]
    for k in range(20):
        mean = np.stack([np.bincount(u, xyz[v, d], len(xyz)) for d in range(3)], 1) / degree
        xyz = xyz + (0.5 if k % 2 == 0 else -0.53) * (mean - xyz)
    return xyz, tri.astype(np.int32)


@functools.lru_cache(maxsize=10)
def _globule(atoms, grid, which=0):
    """A compact heap of atoms with holes and the isosurface of their summed Gaussians."""
    rng = np.random.default_rng(1000 * atoms + which)
    radius = 38.7 * (atoms / 20000) ** (1 / 3)
    m = int(radius / 2.0) + 2
    site = np.stack(np.meshgrid(*[np.arange(-m, m + 1)] * 3, indexing="ij"), -1).reshape(-1, 3) * 2.05
    site = site[np.argsort(np.linalg.norm(site, axis=1) * rng.uniform(0.85, 1.15, len(site)))]
    site = site[: int(1.3 * atoms) + 1]
    site = site[np.sort(rng.permutation(len(site))[:atoms])] + rng.uniform(-0.4, 0.4, (atoms, 3))
    r = rng.uniform(1.2, 2.0, atoms)
    q = rng.normal(0.0, 0.35, atoms)
    low = site.min(0) - 5.2 - 2 * grid
    shape = np.ceil((site.max(0) + 5.2 + 2 * grid - low) / grid).astype(int) + 1
    value = np.full(shape, -1.0)
    for a, ra in zip(site, r):                        # exp(2.3 (1 - d^2 / r^2)), cut off below 1e-4
        lo = np.maximum(np.floor((a - 2.3 * ra - low) / grid).astype(int), 0)
        hi = np.minimum(np.ceil((a + 2.3 * ra - low) / grid).astype(int) + 1, shape)
        e = [np.exp(-2.3 / ra ** 2 * (low[d] + grid * np.arange(lo[d], hi[d]) - a[d]) ** 2) for d in range(3)]
        value[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] += math.exp(2.3) * e[0][:, None, None] * e[1][:, None] * e[2]
    value[np.abs(value) < 1e-9] = 1e-9
    xyz, tri = _outer_and_smooth(*_isosurface(value, low, grid))
    return xyz, tri, site, q - q.mean()


def _rotation(rng):
    q, r = np.linalg.qr(rng.normal(size=(3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


@functools.lru_cache(maxsize=1)
def _cluster(copies, atoms, grid):
    """Turned copies of one globule on a shell, apart from each other."""
    xyz, tri, site, q = _globule(atoms, grid)
    rng = np.random.default_rng(copies)
    reach = max(np.linalg.norm(xyz, axis=1).max(), 1.0)
    k = np.arange(copies) + 0.5
    z, turn = 1 - 2 * k / copies, math.pi * (1 + math.sqrt(5)) * k
    s = np.sqrt(1 - z * z)
    place = np.stack([s * np.cos(turn), s * np.sin(turn), z], 1)
    gap = np.linalg.norm(place[:, None] - place[None], axis=2) + 9 * np.eye(copies)
    place *= 2.05 * reach / gap.min()
    turns = [_rotation(rng) for _ in range(copies)]
    return (np.concatenate([xyz @ t.T + p for t, p in zip(turns, place)]),
            np.concatenate([tri + i * len(xyz) for i in range(copies)]).astype(np.int32),
            np.concatenate([site @ t.T + p for t, p in zip(turns, place)]), np.tile(q, copies))


def _molecule(case, seed, which=0):
    """Node positions, triangles, charge positions and charges of a case, turned as the seed says."""
    rng = np.random.default_rng((seed, which))
    if case["shape"] == "sphere":
        xyz, tri = _sphere(case["freq"] + which)
        xyz = xyz * case["radius"]
        n = case["atoms"]
        site, q = np.zeros((1, 3)), np.ones(1)
        if n > 1:
            site = rng.normal(size=(n, 3))
            site *= (0.8 * case["radius"] * rng.random(n) ** (1 / 3) / np.linalg.norm(site, axis=1))[:, None]
            q = rng.uniform(-1, 1, n)
    elif case["shape"] == "globule":
        xyz, tri, site, q = _globule(case["atoms"] + which, case["grid"], which)
    else:
        xyz, tri, site, q = _cluster(case["copies"], case["atoms"], case["grid"])
    turn = _rotation(rng)
    return xyz @ turn.T, tri, site @ turn.T, q


def _unknowns(xyz, seed):
    """x = [f; h] like a Krylov vector: a smooth field over the surface with some noise."""
    rng = np.random.default_rng((seed, 77))
    c = (xyz - xyz.mean(0)) / np.abs(xyz - xyz.mean(0)).max()
    w = rng.normal(size=(2, 10))
    base = np.stack([np.ones(len(c)), *c.T, *(c * c).T, *(c * np.roll(c, 1, axis=1)).T])
    return ((w @ base).reshape(-1) + 0.2 * rng.normal(size=2 * len(c))).astype(np.float32)


def _nodes(case):
    """About how many nodes a case's molecule has (for work(); a globule's surface is counted from its size)."""
    if case["shape"] == "sphere":
        return 10 * case["freq"] ** 2 + 2
    one = 500 * case["atoms"] ** 0.81 * (0.4 / case["grid"]) ** 2
    return one * case.get("copies", 1)


# ---- one pass -----------------------------------------------------------------------------
@functools.lru_cache(maxsize=1)
def _stream():
    return torch.cuda.Stream()


def _options(case):
    return dict(eps_in=case["eps_in"], eps_out=80.0, kappa=case["kappa"], order=case["order"],
                precision=case["precision"])


def prepare(case, seed):
    use = case["use"]
    if use == "batch":
        mols = [_molecule(case, seed, k) for k in range(case["count"])]
        return dict(use=use, handles=[pb.Handle(*m, **_options(case)) for m in mols])
    mol = _molecule(case, seed)
    if use == "request":
        return dict(use=use, mol=mol, options=_options(case))
    if use == "solve":
        return dict(use=use, handle=pb.Handle(*mol, stream=_stream(), **_options(case)))
    handle = pb.Handle(*mol[:2], stream=_stream(), **_options(case))
    x = torch.from_numpy(_unknowns(mol[0], seed))
    if use == "host":
        return dict(use=use, handle=handle, x=x.pin_memory(), y=torch.empty_like(x).pin_memory())
    x = x.cuda()
    return dict(use=use, handle=handle, x=x, y=torch.empty_like(x))


def run(state):
    use = state["use"]
    if use == "product":
        state["handle"].matvec(state["x"], state["y"])
        return state["y"]
    if use == "host":
        return state["handle"].matvec_host(state["x"], state["y"])
    if use == "solve":
        f, h, _ = state["handle"].solve()
        return dict(f=f, h=h, energy=state["handle"].energy())
    if use == "request":
        with pb.Handle(*state["mol"], **state["options"]) as handle:
            f, h, _ = handle.solve()
            return dict(f=f, h=h, energy=handle.energy())
    solved = pb.solve_batch(state["handles"])
    return [dict(f=f, h=h, energy=handle.energy()) for handle, (f, h, _) in zip(state["handles"], solved)]


def work(case):
    """Of a product: the node data (32 B), x and y (16 B) and the near coefficients (20 B each, 20 or 36 to a node)
    once, 62 operations for each of about 770 point pairs of a node, and the translations.  Of the others: their
    products (8 of them for a solve and its check at the least) and, for a request, the near coefficients'
    quadrature (about 40 points of 60 operations for each)."""
    n = _nodes(case)
    near = 20 if case["shape"] == "sphere" else 36
    expansions = 2 * 2 * 2 * case["order"] ** 3 * 6
    one = dict(bytes=n * (48.0 + 20 * near), flops=n * (62.0 * 770 + 8 * near + expansions))
    times = {"product": 1, "host": 1, "solve": 8, "request": 8, "batch": 8 * case.get("count", 1)}[case["use"]]
    extra = n * near * 2400.0 if case["use"] == "request" else 0.0
    return dict(bytes=one["bytes"] * times, flops=one["flops"] * times + extra)


# ---- the same in 64 bits ------------------------------------------------------------------
class _Exact:
    """The node-patch operator summed over all pairs in FP64 (near pairs by quadrature over the patch)."""

    def __init__(self, case, mol, dense=False):
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.kappa, self.ebar = case["kappa"], 80.0 / case["eps_in"]
        self.alpha = 0.5 / self.ebar + 0.5
        xyz, tri = torch.from_numpy(mol[0]).to(dev), torch.from_numpy(mol[1].astype(np.int64)).to(dev)
        self.xyz, n = xyz, len(mol[0])
        p = xyz[tri]
        cross = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
        length = cross.norm(dim=1)
        self.facet = cross / length[:, None]
        self.area = torch.zeros(n, dtype=xyz.dtype, device=dev)
        normal = torch.zeros_like(xyz)
        self.rho = torch.zeros_like(self.area)
        # the patch of node v in triangle (v, a, b): (v, mid(v, a), centroid) and (v, centroid, mid(v, b))
        piece, owner, facet = [], [], []
        centroid = p.mean(1)
        for k in range(3):
            v, a, b = tri[:, k], (p[:, k] + p[:, (k + 1) % 3]) / 2, (p[:, k] + p[:, (k + 2) % 3]) / 2
            self.area.index_add_(0, v, length / 6)
            normal.index_add_(0, v, cross)
            for q in (a, b, centroid):
                self.rho.scatter_reduce_(0, v, (q - p[:, k]).norm(dim=1), "amax")
            piece += [torch.stack([p[:, k], a, centroid], 1), torch.stack([p[:, k], centroid, b], 1)]
            owner += [v, v]
            facet += [self.facet, self.facet]
        self.normal = normal / normal.norm(dim=1, keepdim=True)
        owner = torch.cat(owner)
        order = torch.argsort(owner, stable=True)
        self.piece, self.piece_normal = torch.cat(piece)[order], torch.cat(facet)[order]
        count = torch.bincount(owner, minlength=n)
        self.piece_end = torch.cumsum(count, 0)
        self.piece_begin = self.piece_end - count
        self._rows = self._dense = None
        self._near()
        if dense:
            self._dense = torch.cat([torch.cat([m for _, m in self._far_rows(top=True)]),
                                     torch.cat([m for _, m in self._far_rows(top=False)])])

    def _kernels(self, r2, ndn, n0d, nn0):
        """Eq. 6's four integrands, without 1 / (4 pi)."""
        ri = torch.rsqrt(r2)
        ri2 = ri * ri
        g3 = ri * ri2
        kr = self.kappa * r2 * ri
        e = torch.exp(-kr)
        e1 = e * (1 + kr)
        e2 = e1 + e * kr * kr / 3
        return (-torch.expm1(-kr) * ri, ndn * g3 * (1 / self.ebar - e1), n0d * g3 * (e1 / self.ebar - 1),
                (nn0 * g3 * (1 - e1) - 3 * ndn * n0d * g3 * ri2 * (1 - e2)) / self.ebar)

    def _near(self):
        """Near pairs, and what is added to their point terms: quadrature minus point rule, and the self patches."""
        n, dev = len(self.xyz), self.xyz.device
        pairs = []
        step = max(1, 30_000_000 // n)
        sq = (self.xyz * self.xyz).sum(1)
        for lo in range(0, n, step):
            x = self.xyz[lo:lo + step]
            r2 = sq[lo:lo + step, None] + sq[None] - 2 * x @ self.xyz.T
            reach = NEAR_C * (self.rho[lo:lo + step, None] + self.rho[None])
            some = torch.nonzero(r2 < reach * reach * (1 + 1e-9) + 1e-9)
            some[:, 0] += lo
            pairs.append(some[some[:, 0] != some[:, 1]])
        pairs = torch.cat(pairs)
        close = (self.xyz[pairs[:, 0]] - self.xyz[pairs[:, 1]]).norm(dim=1)
        pairs = pairs[close < NEAR_C * (self.rho[pairs[:, 0]] + self.rho[pairs[:, 1]])]
        value = torch.zeros(len(pairs), 4, dtype=torch.float64, device=dev)
        for lo in range(0, len(pairs), 200_000):
            value[lo:lo + 200_000] = self._quadrature(pairs[lo:lo + 200_000])
        p, t = pairs.T
        d = self.xyz[p] - self.xyz[t]
        point = torch.stack(self._kernels((d * d).sum(1), (self.normal[t] * d).sum(1), (self.normal[p] * d).sum(1),
                                          (self.normal[t] * self.normal[p]).sum(1)), 1) * self.area[t, None] / (4 * math.pi)
        every = torch.arange(n, device=dev)
        self.rows, self.cols = torch.cat([p, every]), torch.cat([t, every])
        self.coef = torch.cat([value - point, self._self()])

    def _quadrature(self, pairs):
        """Radon's 7-point rule on the source's patch pieces, each split 1 -> 4 (six times at most) while the target is
        closer to its centroid than three times its longest edge."""
        r15 = math.sqrt(15.0)
        a, b = (6 - r15) / 21, (6 + r15) / 21
        bary = torch.tensor([[1 / 3] * 3] + [[c] * k + [1 - 2 * c] + [c] * (2 - k) for c in (a, b) for k in range(3)],
                            dtype=torch.float64, device=pairs.device)
        weight = torch.tensor([9 / 40] + [(155 - r15) / 1200] * 3 + [(155 + r15) / 1200] * 3, dtype=torch.float64,
                              device=pairs.device)
        p, t = pairs.T
        count = self.piece_end[t] - self.piece_begin[t]
        entry = torch.repeat_interleave(torch.arange(len(pairs), device=pairs.device), count)
        index = torch.arange(len(entry), device=pairs.device) - torch.repeat_interleave(torch.cumsum(count, 0) - count, count)
        index += self.piece_begin[t][entry]
        shape = self.piece[index] - self.xyz[p[entry], None]
        source = self.piece_normal[index]
        out = torch.zeros(len(pairs), 4, dtype=torch.float64, device=pairs.device)
        for depth in range(7):
            edge2 = ((shape - shape.roll(1, 1)) ** 2).sum(2).amax(1)
            split = (shape.mean(1) ** 2).sum(1) < 9 * edge2
            if depth == 6:
                split[:] = False
            s, e, ns = shape[~split], entry[~split], source[~split]
            area = torch.linalg.cross(s[:, 1] - s[:, 0], s[:, 2] - s[:, 0]).norm(dim=1) / 2
            d = -(bary @ s)                                        # target minus quadrature point
            n0 = self.normal[p[e]]
            k = self._kernels((d * d).sum(2), (d * ns[:, None]).sum(2), (d * n0[:, None]).sum(2),
                              (ns * n0).sum(1, keepdim=True))
            out.index_add_(0, e, torch.stack([(v @ weight) * area for v in k], 1) / (4 * math.pi))
            s, entry, source = shape[split], entry[split], source[split]
            if not len(s):
                break
            ab, bc, ca = ((s[:, i] + s[:, (i + 1) % 3]) / 2 for i in range(3))
            shape = torch.cat([torch.stack(c, 1) for c in ((s[:, 0], ab, ca), (ab, s[:, 1], bc), (ca, bc, s[:, 2]), (ab, bc, ca))])
            entry, source = entry.repeat(4), source.repeat(4, 1)
        return out

    def _self(self):
        """The patch of a node on its own tangent plane, in polar coordinates about it, 16 x 16 Gauss points."""
        x, w = (torch.from_numpy(v).to(self.xyz.device) for v in np.polynomial.legendre.leggauss(16))
        x, w = (x + 1) / 2, w / 2
        n = len(self.xyz)
        node = torch.repeat_interleave(torch.arange(n, device=x.device), self.piece_end - self.piece_begin)
        out = torch.zeros(n, 4, dtype=torch.float64, device=x.device)
        for lo in range(0, len(node), 100_000):
            at = node[lo:lo + 100_000]
            e = self.piece[lo:lo + 100_000, 1:] - self.xyz[at, None]
            n0 = self.normal[at, None]
            e = e - (e * n0).sum(2, keepdim=True) * n0
            jac = torch.linalg.cross(e[:, 0], e[:, 1]).norm(dim=1)[:, None]
            far = (e[:, 0, None] + x[:, None] * (e[:, 1] - e[:, 0])[:, None]).norm(dim=2)
            kr = self.kappa * far[..., None] * x
            small = kr < 1e-3                                      # 1 - e^-x (1 + x) without cancellation
            p1 = torch.where(small, kr * kr * (0.5 - kr / 3 + kr * kr / 8), -torch.expm1(-kr) - kr * torch.exp(-kr))
            a = ((-torch.expm1(-kr)) @ w / far * jac) @ w
            d = (p1 @ (w / x ** 2) / far ** 3 * jac) @ w
            zero = torch.zeros_like(a)
            out.index_add_(0, at, torch.stack([a, zero, zero, d / self.ebar], 1) / (4 * math.pi))
        return out

    def _point_rows(self, step):
        n = len(self.xyz)
        sq, yn = (self.xyz * self.xyz).sum(1), (self.xyz * self.normal).sum(1)
        for lo in range(0, n, step):
            x, n0 = self.xyz[lo:lo + step], self.normal[lo:lo + step]
            r2 = torch.addmm(sq[lo:lo + step, None] + sq[None], x, self.xyz.T, alpha=-2)
            row = torch.arange(len(x), device=x.device)
            r2[row, row + lo] = 1e30                               # no point term of a node at itself
            k = self._kernels(r2, x @ self.normal.T - yn[None], (x * n0).sum(1, keepdim=True) - n0 @ self.xyz.T,
                              n0 @ self.normal.T)
            for v in k:
                v[row, row + lo] = 0.0
            yield lo, k

    def _far_rows(self, top):
        n = len(self.xyz)
        c = self.area[None] / (4 * math.pi)
        for lo, (ka, kb, kc, kd) in self._point_rows(max(1, 4_000_000 // n)):
            left, right = (kb * c, -ka * c) if top else (kd * c, -kc * c)
            m = len(left)
            some = (self.rows >= lo) & (self.rows < lo + m)
            r, t, v = self.rows[some] - lo, self.cols[some], self.coef[some]
            left.index_put_((r, t), v[:, 1] if top else v[:, 3], accumulate=True)
            right.index_put_((r, t), -(v[:, 0] if top else v[:, 2]), accumulate=True)
            row = torch.arange(m, device=left.device)
            (left if top else right)[row, row + lo] += self.alpha
            yield lo, torch.cat([left, right], 1)

    def product(self, x):
        if self._dense is not None:
            return self._dense @ x
        n = len(self.xyz)
        f, h = x[:n], x[n:]
        y = self.alpha * x
        af, ah = (v * self.area / (4 * math.pi) for v in (f, h))
        for lo, (ka, kb, kc, kd) in self._point_rows(max(1, 4_000_000 // n)):
            y[lo:lo + len(ka)] += kb @ af - ka @ ah
            y[n + lo:n + lo + len(ka)] += kd @ af - kc @ ah
        v, t = self.coef, self.cols
        y.index_add_(0, self.rows, v[:, 1] * f[t] - v[:, 0] * h[t])
        y.index_add_(0, n + self.rows, v[:, 3] * f[t] - v[:, 2] * h[t])
        return y

    def solve(self, site, q):
        """f, h and the solvation energy: Arnoldi steps on the dense operator to 1e-11."""
        site, q = (torch.from_numpy(v).to(self.xyz.device) for v in (site, q))
        d = self.xyz[:, None] - site[None]
        g = (d * d).sum(2).rsqrt()
        b = torch.cat([g @ q, -(g ** 3 * (d * self.normal[:, None]).sum(2)) @ q]) / (4 * math.pi * 80.0)
        basis, hess, beta = [b / b.norm()], np.zeros((202, 201)), float(b.norm())
        for j in range(200):
            w = self.product(basis[j])
            v = torch.stack(basis)
            for _ in range(2):
                c = v @ w
                w = w - c @ v
                hess[: j + 1, j] += c.cpu().numpy()
            hess[j + 1, j] = float(w.norm())
            basis.append(w / w.norm())
            rhs = np.zeros(j + 2)
            rhs[0] = beta
            y, *_ = np.linalg.lstsq(hess[: j + 2, : j + 1], rhs, rcond=None)
            if np.linalg.norm(rhs - hess[: j + 2, : j + 1] @ y) < 1e-11 * beta:
                break
        x = torch.from_numpy(y).to(b.device) @ torch.stack(basis[: j + 1])
        n = len(self.xyz)
        f, h = x[:n], x[n:]
        # the reaction field at the charges, from the surface
        phi = (self.ebar * self.area * h) @ g + (self.area * f) @ (g ** 3 * (d * self.normal[:, None]).sum(2))
        return dict(f=f, h=h, energy=torch.tensor(0.5 * COULOMB * float(phi @ q), dtype=torch.float64))


def exact(case, seed):
    use = case["use"]
    if case["shape"] == "cluster":
        return None
    if use == "batch":
        mols = [_molecule(case, seed, k) for k in range(case["count"])]
        if sum(len(m[0]) for m in mols) > 8 * EXACT_DENSE:
            return None
        return [_Exact(case, m, dense=True).solve(*m[2:]) if len(m[0]) <= EXACT_DENSE else dict(f=None, h=None, energy=None)
                for m in mols]
    mol = _molecule(case, seed)
    if len(mol[0]) > (EXACT_NODES if use in ("product", "host") else EXACT_DENSE):
        return None
    if use in ("product", "host"):
        e = _Exact(case, mol)
        return e.product(torch.from_numpy(_unknowns(mol[0], seed)).to(e.xyz.device).double())
    return _Exact(case, mol, dense=True).solve(*mol[2:])
