"""The far-field passes against the sums they compute: list 2 and list 4 by interpolation on the
handle's own tree, everything else point by point, restated in float64.  Interpolation error is
in both, so what is left is rounding, and a lost weight, leaf or node shows at any order."""
import numpy as np
import pytest

import oracle
import synthetic
from test_near_setup import globe
from test_p2p_pairs import EPS, far_parts, whole_matrix

pytestmark = pytest.mark.gpu


def basis(n, x):
    """The n interpolation polynomials of the Chebyshev points and their derivatives at x."""
    k = np.arange(n)
    pts = np.cos((2 * k + 1) * np.pi / (2 * n))
    T, dT = np.ones(x.shape + (n,)), np.zeros(x.shape + (n,))
    T[..., 1], dT[..., 1] = x, 1.0
    for j in range(2, n):
        T[..., j] = 2 * x * T[..., j - 1] - T[..., j - 2]
        dT[..., j] = 2 * T[..., j - 1] + 2 * x * dT[..., j - 1] - dT[..., j - 2]
    C = np.cos(k[None] * np.arccos(pts)[:, None]) * np.where(k == 0, 1.0, 2.0) / n
    return T @ C.T, dT @ C.T, pts


def weights(n, x, nrm, center, w):
    """S and n . grad S of a box's n^3 points at its nodes."""
    S, D, pts = basis(n, (x - center) / w)
    cube = lambda a, b, c: np.einsum("ti,tj,tk->tijk", a, b, c).reshape(len(x), -1)
    s = [S[:, d] for d in range(3)]
    g = [D[:, d] / w for d in range(3)]
    grad = (nrm[:, :1] * cube(g[0], s[1], s[2]) + nrm[:, 1:2] * cube(s[0], g[1], s[2]) + nrm[:, 2:] * cube(s[0], s[1], g[2]))
    nodes = np.stack(np.meshgrid(pts, pts, pts, indexing="ij"), -1).reshape(-1, 3) * w + center
    return cube(*s), grad, nodes


def kernels(a, b, kappa):
    r = np.linalg.norm(a[:, None] - b[None], axis=2)
    G = 1 / (4 * np.pi * r)
    return G, G * np.exp(-kappa * r)


def point_kernels(x, n0, y, n1, kappa):
    """(K, dK/dn_y, dK/dn_x, d2K/dn_x dn_y) of both kernels between points (zero where they meet)."""
    d = x[:, None] - y[None]
    r = np.sqrt((d * d).sum(2))
    meet = r == 0
    r[meet] = 1.0
    ny, nx, nn = (d * n1[None]).sum(2), (d * n0[:, None]).sum(2), n0 @ n1.T
    out = []
    for k in (0.0, kappa):
        e = np.where(meet, 0.0, np.exp(-k * r) / (4 * np.pi))
        e1, e2 = e * (1 + k * r), e * (1 + k * r + (k * r) ** 2 / 3)
        out.append((e / r, e1 * ny / r ** 3, -e1 * nx / r ** 3, e1 * nn / r ** 3 - 3 * e2 * nx * ny / r ** 5))
    return out


def restated(h, mol, o, x, order):
    """The far part of the product, its terms' magnitudes, and the number of list-4 boxes that
    are taken by interpolation."""
    n, kappa, ebar = mol.n_nodes, mol.kappa, mol.eps_out / mol.eps_in
    area, nrm, _ = o.geometry()
    t = h.tree()
    perm, rng, level = t["perm"], t["range"], t["level"]
    lo, hi = mol.xyz.min(0), mol.xyz.max(0)
    w0 = 0.5 * (hi - lo).max() * (1 + 1e-6)
    w = w0 / 2.0 ** level
    center = 0.5 * (lo + hi) - w0 + (2 * t["anchor"] + 1) * w[:, None]
    nodes_of = lambda b: perm[rng[b, 0]:rng[b, 1]]
    cache = {}

    def box(b):
        if b not in cache:
            i = nodes_of(b)
            cache[b] = (i, *weights(order, mol.xyz[i], nrm[i], center[b], w[b]))
        return cache[b]

    f, hh = x[:n] * area, x[n:] * area
    y, mag, used, p2l = np.zeros(2 * n), np.zeros(2 * n), np.zeros((n, n), np.int8), 0

    def add(i, j, blocks, mags):
        (G, Gy, Gx, Gxy), (u, uy, ux, uxy) = blocks
        y[i] += (Gy / ebar - uy) @ f[j] - (G - u) @ hh[j]
        y[n + i] += ((Gxy - uxy) / ebar) @ f[j] - (Gx - ux / ebar) @ hh[j]
        (G, Gy, Gx, Gxy), (u, uy, ux, uxy) = mags
        mag[i] += (Gy / ebar + uy) @ np.abs(f[j]) + (G + u) @ np.abs(hh[j])
        mag[n + i] += ((Gxy + uxy) / ebar) @ np.abs(f[j]) + (Gx + ux / ebar) @ np.abs(hh[j])
        used[np.ix_(i, j)] += 1

    def through(St, dSt, K, Sc, dSc):
        return [(St @ k @ Sc.T, St @ k @ dSc.T, dSt @ k @ Sc.T, dSt @ k @ dSc.T) for k in K]

    for b in range(len(level)):
        for c in t["v_idx"][t["v_ptr"][b]:t["v_ptr"][b + 1]]:
            i, St, dSt, at = box(b)
            j, Sc, dSc, ac = box(c)
            K = kernels(at, ac, kappa)
            add(i, j, through(St, dSt, K, Sc, dSc), through(*map(np.abs, (St, dSt)), K, *map(np.abs, (Sc, dSc))))
        i = nodes_of(b)
        for c in t["x_idx"][t["x_ptr"][b]:t["x_ptr"][b + 1]]:
            j = nodes_of(c)
            if len(i) <= order ** 3:
                continue                                     # summed directly, below
            p2l += 1
            _, St, dSt, at = box(b)
            P = point_kernels(at, np.zeros_like(at), mol.xyz[j], nrm[j], kappa)
            block = lambda A, dA, q: [(A @ k[0], A @ k[1], dA @ k[0], dA @ k[1]) for k in q]
            add(i, j, block(St, dSt, P), block(np.abs(St), np.abs(dSt), [[np.abs(v) for v in k] for k in P]))
    rest = (used == 0) & ~whole_matrix(h)
    np.fill_diagonal(rest, False)
    P = [tuple(np.where(rest, v, 0) for v in k) for k in point_kernels(mol.xyz, nrm, mol.xyz, nrm, kappa)]
    assert used.max() == 1
    everyone = np.arange(n)
    add(everyone, everyone, P, [tuple(np.abs(v) for v in k) for k in P])
    return y, mag, p2l


def mesh(kind, seed):
    if kind == "globe":
        return globe(14, 40, seed)
    mol = synthetic.born_ion(subdiv=int(kind[-1]))
    rng = np.random.default_rng(seed)
    mol.xyz = mol.xyz * (1 + 0.02 * rng.standard_normal((mol.n_nodes, 1)))
    return mol


CASES = [("sphere 2", 1, order, 0) for order in (2, 3, 4, 5, 6)] + [("sphere 3", 30, order, 0) for order in range(2, 9)]
CASES += [("globe", 12, 2, 0), ("globe", 12, 3, 0), ("globe", 24, 4, 0), ("globe", 24, 5, 0)]
CASES += [("sphere 2", 1, 2, 1), ("sphere 2", 1, 4, 1), ("sphere 3", 30, 6, 1), ("globe", 12, 2, 1), ("globe", 24, 4, 1)]


@pytest.mark.parametrize("kind,leaf_cap,order,precision", CASES)
def test_far_part_equals_its_sums(kind, leaf_cap, order, precision):
    """Each of a box's n^3 polynomials is a product of three Chebyshev sums of n terms up to 2,
    so their rounding comes to 6 (n + 2) n^3 units of the magnitudes on either side of a
    translation, n times that in the normal derivative; operators compressed at 1e-5 and split
    into BF16 pairs get the product's 1e-4."""
    import paper_1710_06316_gb300 as pb
    mol = mesh(kind, order)
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.random_unknowns(mol.n_nodes, order).astype(np.float32).astype(np.float64)
    options = dict(m2l_tol=-1.0) if precision == 0 else {}
    with pb.Handle.for_molecule(mol, order=order, leaf_cap=leaf_cap, precision=precision, **options) as h:
        assert h.info()["n_m2l_pairs"] > 0
        y = far_parts(h, x)
        ref, mag, p2l = restated(h, mol, o, x, order)
    assert p2l > 0 or (kind, order) != ("globe", 2)          # list 4 through local expansions
    n = mol.n_nodes
    bar = EPS * 12 * (order + 2) * order ** 3 + (1e-4 if precision else 0.0)
    err = np.abs(y - ref) / mag
    assert err[:n].max() <= bar and err[n:].max() <= order * bar, (err[:n].max() / bar, err[n:].max() / (order * bar))
