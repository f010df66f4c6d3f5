"""The far-field passes on both sides of the lines where their kernels change form: L2P with the
leaves of a block staged or read where they lie (six leaves), P2M with a warp to a leaf or to
several (odd orders, by the number of leaves), FP32 translations beside P2P and after it.  Rows of
the far part against their own sums in float64."""
import numpy as np
import pytest

import oracle
import synthetic
from test_far_interpolation import kernels, point_kernels, weights
from test_p2p_pairs import EPS, far_parts, whole_matrix

pytestmark = pytest.mark.gpu


def leaves_of(t):
    n = len(t["level"])
    parent = np.zeros(n, bool)
    parent[t["parent"][t["parent"] >= 0]] = True
    return np.flatnonzero(~parent)


def block_spans(t, n, nodes=128):
    """Leaves that each block of 128 nodes (Morton order) spans."""
    leaf = np.zeros(n, np.int64)
    order = leaves_of(t)
    order = order[np.argsort(t["range"][order, 0])]
    for k, b in enumerate(order):
        leaf[t["range"][b, 0]:t["range"][b, 1]] = k
    return np.array([leaf[min(n, i + nodes) - 1] - leaf[i] + 1 for i in range(0, n, nodes)])


def rows_of(h, mol, o, x, order, rows):
    """The far part at `rows` and its terms' magnitudes (list 4 summed directly)."""
    n, kappa, ebar = mol.n_nodes, mol.kappa, mol.eps_out / mol.eps_in
    area, nrm, _ = o.geometry()
    t = h.tree()
    lo, hi = mol.xyz.min(0), mol.xyz.max(0)
    w0 = 0.5 * (hi - lo).max() * (1 + 1e-6)
    w = w0 / 2.0 ** t["level"]
    center = 0.5 * (lo + hi) - w0 + (2 * t["anchor"] + 1) * w[:, None]
    nodes_of = lambda b: t["perm"][t["range"][b, 0]:t["range"][b, 1]]
    f, hh = x[:n] * area, x[n:] * area
    rp, col, _, whole = h.near()
    place = np.empty(n, np.int64)
    place[t["perm"]] = np.arange(n)
    y, mag = np.zeros((2, len(rows))), np.zeros((2, len(rows)))
    for k, r in enumerate(rows):
        xr, nr = mol.xyz[r:r + 1], nrm[r:r + 1]
        direct = np.ones(n, bool)
        direct[r] = False
        direct[col[rp[r]:rp[r + 1]][whole[rp[r]:rp[r + 1]]]] = False

        def add(j, blocks, size):
            for out, sgn, q in ((y, 1, blocks), (mag, 0, size)):
                (G, Gy, Gx, Gxy), (u, uy, ux, uxy) = q
                a, b = (f[j], hh[j]) if sgn else (np.abs(f[j]), np.abs(hh[j]))
                m = -1 if sgn else 1
                out[0, k] += ((Gy / ebar + m * uy) @ a + m * (G + m * u) @ b)[0]
                out[1, k] += ((Gxy + m * uxy) / ebar @ a + m * (Gx + m * ux / ebar) @ b)[0]

        for b in np.flatnonzero((t["range"][:, 0] <= place[r]) & (place[r] < t["range"][:, 1])):
            St, dSt, at = weights(order, xr, nr, center[b], w[b])
            for c in t["v_idx"][t["v_ptr"][b]:t["v_ptr"][b + 1]]:
                j = nodes_of(c)
                Sc, dSc, ac = weights(order, mol.xyz[j], nrm[j], center[c], w[c])
                K = kernels(at, ac, kappa)
                through = lambda A, dA, B, dB: [(A @ q @ B.T, A @ q @ dB.T, dA @ q @ B.T, dA @ q @ dB.T) for q in K]
                add(j, through(St, dSt, Sc, dSc), through(*map(np.abs, (St, dSt, Sc, dSc))))
                direct[j] = False
            assert t["x_ptr"][b] == t["x_ptr"][b + 1] or len(nodes_of(b)) <= order ** 3
        j = np.flatnonzero(direct)
        P = point_kernels(xr, nr, mol.xyz[j], nrm[j], kappa)
        add(j, P, [tuple(np.abs(v) for v in q) for q in P])
    return y.reshape(-1), mag.reshape(-1)


def check(mol, order, leaf_cap, seed):
    import paper_1710_06316_gb300 as pb
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.random_unknowns(mol.n_nodes, seed).astype(np.float32).astype(np.float64)
    with pb.Handle.for_molecule(mol, order=order, leaf_cap=leaf_cap, m2l_tol=-1.0) as h:
        assert h.info()["n_m2l_pairs"] > 0
        y = far_parts(h, x).reshape(2, -1)
        rows = np.sort(np.random.default_rng(seed).choice(mol.n_nodes, 24, replace=False))
        ref, mag = rows_of(h, mol, o, x, order, rows)
        t = h.tree()
    err = np.abs(y[:, rows].reshape(-1) - ref) / mag
    bar = EPS * 12 * (order + 2) * order ** 3            # as in test_far_interpolation
    assert err[:24].max() <= bar and err[24:].max() <= order * bar, err.max() / bar
    return t


def sphere(subdiv, seed):
    mol = synthetic.born_ion(subdiv=subdiv)
    rng = np.random.default_rng(seed)
    mol.xyz = mol.xyz * (1 + 0.01 * rng.standard_normal((mol.n_nodes, 1)))
    return mol


@pytest.mark.parametrize("order,leaf_cap", [(3, 90), (4, 90), (6, 90), (4, 58), (5, 58), (6, 58), (3, 2), (8, 12)])
def test_blocks_of_few_and_of_many_leaves(order, leaf_cap):
    mol = sphere(4, order)
    spans = block_spans(check(mol, order, leaf_cap, leaf_cap), mol.n_nodes)[:-1]   # whole blocks
    if leaf_cap == 90:
        assert (spans <= 6).all()
    elif leaf_cap == 58:
        assert (spans <= 6).any() and (spans > 6).any()
    else:
        assert (spans > 6).all()


@pytest.mark.parametrize("order,leaves_per_warp", [(3, 5), (5, 3), (7, 2)])
def test_many_leaves_at_odd_orders(order, leaves_per_warp):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mol = sphere(5, order)
    t = check(mol, order, 1, order)
    assert len(leaves_of(t)) > 12 * leaves_per_warp * sms


def test_translations_after_p2p():
    """Order 4 in FP32 on a mesh of small leaves: two translations or more to 1000 pairs."""
    mol = sphere(4, 1)
    check(mol, 4, 8, 3)
    import paper_1710_06316_gb300 as pb
    with pb.Handle.for_molecule(mol, order=4, leaf_cap=8) as h:
        assert 500 * h.info()["n_m2l_pairs"] >= h.info()["n_p2p_pairs"]
