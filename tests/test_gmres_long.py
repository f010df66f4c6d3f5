"""The Arnoldi step's kernels at their edges: vectors of less than a tile, of a tile and a bit,
cycles longer than the shared-memory forms of the Givens update and the back substitution.
Bar: the solution's 1e-4 against the oracle's solve."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


def check(subdiv, restart, tol, max_restart):
    import paper_1710_06316_gb300 as pb
    mol = synthetic.kirkwood_sphere(subdiv=subdiv, radius=6.0, n_charges=5, r_charges=4.0)
    ref = oracle.Oracle.for_molecule(mol).solve(mol.atoms, mol.q, rel_tol=1e-9)
    with pb.Handle.for_molecule(mol, order=6, tol=tol, restart=restart, max_restart=max_restart) as h:
        f, hh, info = h.solve(raise_on_noconv=False)
        energy = h.energy()
    for a, b in ((f, ref["f"]), (hh, ref["h"])):
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
    assert abs(energy / ref["energy"] - 1) <= 1e-4
    return info["iters"]


@pytest.mark.parametrize("subdiv,restart,max_restart", [(1, 8, 5), (2, 3, 20), (3, 80, 5)])
def test_solution_at_vector_edges(subdiv, restart, max_restart):
    check(subdiv, restart, 1e-6, max_restart)


@pytest.mark.parametrize("restart", [73, 290])
def test_solution_after_long_cycles(restart):
    """The residual estimate falls by about 20 a step on this problem, so a tolerance near the
    smallest double keeps the cycle going past the 72 steps that the back substitution stages."""
    assert check(3, restart, 1e-290, 1) > 72
