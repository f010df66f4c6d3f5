"""Near coefficients where a warp's batches of entries are ragged: poles of many triangles (more
pieces to one entry than a warp reads at a time, thin triangles that split deep), a few nodes
only, and entry counts that are no multiple of a batch.  Reference: the float64 oracle."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


def globe(rings, sides, seed):
    """A closed sphere-like mesh: `rings` circles of `sides` nodes between two poles."""
    rng = np.random.default_rng(seed)
    th = np.pi * (np.arange(rings) + 1) / (rings + 1)
    ph = 2 * np.pi * np.arange(sides) / sides
    ring = np.stack([np.outer(np.sin(th), np.cos(ph)), np.outer(np.sin(th), np.sin(ph)),
                     np.outer(np.cos(th), np.ones(sides))], -1).reshape(-1, 3)
    xyz = np.concatenate([[[0, 0, 1]], ring, [[0, 0, -1]]]) * 2.0
    xyz *= 1 + 0.005 * rng.standard_normal((len(xyz), 1))
    at = lambda r, k: 1 + r * sides + k % sides
    tri = [(0, at(0, k), at(0, k + 1)) for k in range(sides)]
    for r in range(rings - 1):
        for k in range(sides):
            a, b, c, d = at(r, k), at(r, k + 1), at(r + 1, k), at(r + 1, k + 1)
            tri += [(a, c, d), (a, d, b)]
    tri += [(len(xyz) - 1, at(rings - 1, k + 1), at(rings - 1, k)) for k in range(sides)]
    return synthetic.Molecule("globe", xyz, np.array(tri, np.int32), np.zeros((1, 3)), np.ones(1), 2.0, 78.5, 0.104, {})


@pytest.mark.parametrize("rings,sides", [(1, 3), (2, 4), (5, 9), (7, 17), (9, 40), (21, 75)])
def test_near_coefficients_with_ragged_batches(rings, sides):
    """Bars as for any mesh with thin triangles: 1e-5 of the largest coefficient (rounding of
    FP32 sums over up to ~1e4 points), 1e-4 for the single-layer block."""
    import paper_1710_06316_gb300 as pb
    mol = globe(rings, sides, rings)
    o = oracle.Oracle.for_molecule(mol)
    with pb.Handle.for_molecule(mol, order=4, leaf_cap=16) as h:
        rp, col, coef, whole = h.near()
    rp0, col0, _ = o.near_csr()
    assert np.array_equal(rp, rp0)
    for p in range(mol.n_nodes):
        assert np.array_equal(np.sort(col[rp[p]:rp[p + 1]]), col0[rp0[p]:rp0[p + 1]]), p
    rows = np.repeat(np.arange(mol.n_nodes), np.diff(rp))
    near = o.coeffs(rows, col, rule=o.NEAR)
    ref = np.where(whole[:, None], near, near - o.coeffs(rows, col, rule=o.FAR))
    err = np.abs(coef - ref).max(axis=0) / np.abs(ref).max(axis=0)
    assert err[0] < 1e-4 and err[1:].max() < 1e-5, err
