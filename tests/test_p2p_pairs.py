"""The point-to-point pass at the edges of its forms: tested and untested source boxes, with
and without salt, odd source counts, leaves of several source chunks and target tiles, and
source lists longer than one batch of boxes.  Reference: the far-rule pair terms in float64."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def far_parts(h, x):
    import torch
    xd = torch.tensor(x.astype(np.float32), device="cuda")
    yd = torch.empty_like(xd)
    h.matvec_parts(xd, yd, 2)
    torch.cuda.synchronize()
    return yd.cpu().numpy().astype(np.float64)


def pair_sums(mol, o, whole, x):
    """Sums of the far-rule terms over every pair but `whole`, and a rounding bound for each."""
    n, kappa, ebar = mol.n_nodes, mol.kappa, mol.eps_out / mol.eps_in
    area, nrm, _ = o.geometry()
    f, hh = x[:n], x[n:]
    d = mol.xyz[:, None] - mol.xyz[None]
    r2 = (d * d).sum(2)
    use = ~whole
    np.fill_diagonal(use, False)
    r2[~use] = 1.0
    r = np.sqrt(r2)
    ndn, n0d, nn0 = (d * nrm[None]).sum(2), (d * nrm[:, None]).sum(2), nrm @ nrm.T
    G, G3 = 1 / r, 1 / r ** 3
    e = np.exp(-kappa * r)
    e1, e2 = e * (1 + kappa * r), e * (1 + kappa * r + (kappa * r) ** 2 / 3)
    a = area[None] / (4 * np.pi) * use
    y1 = [(f * a * ndn * G3 / ebar), -(f * a * ndn * G3 * e1), -(hh * a * G), (hh * a * G * e)]
    y2 = [f * a * nn0 * G3 / ebar, -3 * f * a * ndn * n0d * G3 / r2 / ebar, -f * a * nn0 * G3 * e1 / ebar,
          3 * f * a * ndn * n0d * G3 / r2 * e2 / ebar, hh * a * n0d * G3, -hh * a * n0d * G3 * e1 / ebar]
    # bounds: 48 operations to a term, and positions rounded about their leaf's centre, whose
    # error counts five times (1/r^5) relative to the pair's distance; |n.d| is rounded as |d|
    c = np.abs(mol.xyz - mol.xyz.mean(0)).max()
    eps = EPS * (48 + 20 * c / r)
    mag1 = np.abs(f) * a * r * G3 * (1 / ebar + e1) + np.abs(hh) * a * G * (1 + e)
    mag2 = np.abs(f) * a * 4 * G3 * (1 + e2) / ebar + np.abs(hh) * a * r * G3 * (1 + e1 / ebar)
    return (np.concatenate([sum(y1).sum(1), sum(y2).sum(1)]),
            np.concatenate([(eps * mag1).sum(1), (eps * mag2).sum(1)]))


def whole_matrix(h):
    rp, col, _, whole = h.near()
    m = np.zeros((h.n, h.n), bool)
    rows = np.repeat(np.arange(h.n), np.diff(rp))
    m[rows[whole], col[whole]] = True
    return m


@pytest.mark.parametrize("kappa", [0.0, 1e-7, 0.104, 3.0])
@pytest.mark.parametrize("subdiv,leaf_cap", [(2, 4096), (3, 4096), (2, 81), (1, 4096)])
def test_pairs_without_far_field(subdiv, leaf_cap, kappa):
    """One leaf (162 nodes: two targets a thread; 642: several target tiles), or a few leaves
    that all touch, so that every pair is P2P's: all sums within their rounding bound."""
    import paper_1710_06316_gb300 as pb
    mol = synthetic.born_ion(subdiv=subdiv, kappa=kappa)
    rng = np.random.default_rng(subdiv)
    mol.xyz = mol.xyz * (1 + 0.05 * rng.standard_normal((mol.n_nodes, 1)) / 2 ** subdiv)
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.random_unknowns(mol.n_nodes, 3).astype(np.float32).astype(np.float64)
    with pb.Handle.for_molecule(mol, order=6, leaf_cap=leaf_cap) as h:
        assert h.info()["n_m2l_pairs"] == 0
        y = far_parts(h, x)
        ref, bound = pair_sums(mol, o, whole_matrix(h), x)
    assert np.all(np.isfinite(y))
    assert np.all(np.abs(y - ref) <= bound), np.max(np.abs(y - ref) / bound)


@pytest.mark.parametrize("near_c", [0.25, 2.0, 6.0])
@pytest.mark.parametrize("leaf_cap", [3, 11])
def test_pairs_of_many_small_boxes(leaf_cap, near_c):
    """Small odd leaves: source lists of more than 64 boxes, and a skip radius from far below
    to far above a leaf's size (hardly any box tested, every box tested).  The bar is the
    product's."""
    import paper_1710_06316_gb300 as pb
    mol = synthetic.born_ion(subdiv=3)
    rng = np.random.default_rng(leaf_cap)
    mol.xyz = mol.xyz * (1 + 0.01 * rng.standard_normal((mol.n_nodes, 1)))
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.random_unknowns(mol.n_nodes, 5).astype(np.float32).astype(np.float64)
    with pb.Handle.for_molecule(mol, order=8, leaf_cap=leaf_cap, near_c=near_c, m2l_tol=-1.0) as h:
        y = far_parts(h, x)
        ref, _ = pair_sums(mol, o, whole_matrix(h), x)
    assert np.linalg.norm(y - ref) <= 1e-4 * np.linalg.norm(ref)
