"""The point-to-point sums away from a solvated protein's constants: dielectric contrast below
one (a droplet of the polar medium), and complete screening.  Reference: the pair terms in
float64, each with its own rounding bound, so that an error that grows with the contrast
shows."""
import numpy as np
import pytest

import oracle
import synthetic
from test_p2p_pairs import EPS, far_parts, pair_sums, whole_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("only", ["h", "both"])
@pytest.mark.parametrize("kappa", [0.0, 0.104, 20.0])
@pytest.mark.parametrize("eps_out", [2.0, 0.008])
def test_pairs_at_low_contrast(eps_out, kappa, only):
    """eps_in 80: the sums stay within the rounding of their terms, also where the screened
    terms, which carry a factor eps_in / eps_out, have died out and do not hide the others."""
    import paper_1710_06316_gb300 as pb
    mol = synthetic.born_ion(subdiv=2, eps_in=80.0, eps_out=eps_out, kappa=kappa)
    rng = np.random.default_rng(7)
    mol.xyz = mol.xyz * (1 + 0.01 * rng.standard_normal((mol.n_nodes, 1)))
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.random_unknowns(mol.n_nodes, 9).astype(np.float32).astype(np.float64)
    if only == "h":
        x[:mol.n_nodes] = 0.0
    with pb.Handle.for_molecule(mol, order=4, leaf_cap=4096) as h:
        y = far_parts(h, x)
        ref, bound = pair_sums(mol, o, whole_matrix(h), x)
    assert np.all(np.abs(y - ref) <= bound), np.max(np.abs(y - ref) / bound)


@pytest.mark.parametrize("eps_out", [2.0, 0.008])
def test_charge_sums_at_low_contrast(eps_out):
    """The charge FMM's right-hand side over one leaf (points only, no interpolation)."""
    import paper_1710_06316_gb300 as pb
    mol = synthetic.kirkwood_sphere(subdiv=2, radius=6.0, n_charges=40, r_charges=4.0, eps_in=80.0, eps_out=eps_out)
    o = oracle.Oracle.for_molecule(mol)
    ref = o.rhs(mol.atoms, mol.q)
    with pb.Handle.for_molecule(mol, order=4, leaf_cap=4096, charge_fmm=2) as h:
        assert h.info()["charge_fmm"] == 1
        b = h.rhs()
    r = np.linalg.norm(mol.xyz[:, None] - mol.atoms[None], axis=2)
    eps = EPS * (48 + 20 * np.abs(mol.xyz).max() / r)          # as in pair_sums
    q = np.abs(mol.q) / (4 * np.pi * eps_out)
    bound = np.concatenate([(eps * q / r).sum(1), (eps * q / r ** 2).sum(1)])
    assert np.all(np.abs(b - ref) <= bound), np.max(np.abs(b - ref) / bound)

@pytest.mark.parametrize("kappa,radius", [(1e20, 2.0), (1e20, 2000.0), (1e12, 2e4), (50.0, 2.0)])
def test_pairs_at_complete_screening(kappa, radius):
    """Screening lengths far below every distance (the limit of a conducting solvent): the
    screened sums vanish, whatever the mesh's unit."""
    import paper_1710_06316_gb300 as pb
    mol = synthetic.born_ion(subdiv=2, radius=radius, kappa=kappa)
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.random_unknowns(mol.n_nodes, 4).astype(np.float32).astype(np.float64)
    with pb.Handle.for_molecule(mol, order=4, leaf_cap=4096) as h:
        y = far_parts(h, x)
        ref, bound = pair_sums(mol, o, whole_matrix(h), x)
    assert np.all(np.isfinite(y))
    assert np.all(np.abs(y - ref) <= bound), np.max(np.abs(y - ref) / bound)
