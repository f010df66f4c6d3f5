"""The far-field passes (P2M, M2M, M2L, L2L, L2P) at every order, odd and even, over leaves of
one to a few nodes (more leaves to a block of nodes than its shared memory holds) and over
ordinary ones, in both precisions.  Reference: the far-rule pair terms in float64."""
import numpy as np
import pytest

import oracle
import synthetic
from test_p2p_pairs import far_parts, pair_sums, whole_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("leaf_cap", [1, 30])
@pytest.mark.parametrize("order", [2, 3, 4, 5, 6, 7, 8])
def test_far_field_at_every_order(order, leaf_cap, precision):
    """The kernels of list-2 and list-4 boxes are interpolated on [-1, 1] with their nearest
    singularity at 3, so an order-n sum converges like rho^-n, rho = 3 + sqrt(8); its normal
    derivative, whose basis functions grow by n^2, like n^2 rho^-n.  The bar takes one order
    off for the three dimensions and two ends of a translation."""
    import paper_1710_06316_gb300 as pb
    mol = synthetic.born_ion(subdiv=3)
    rng = np.random.default_rng(order)
    mol.xyz = mol.xyz * (1 + 0.02 * rng.standard_normal((mol.n_nodes, 1)))
    o = oracle.Oracle.for_molecule(mol)
    x = synthetic.smooth_unknowns(mol.xyz, order).astype(np.float32).astype(np.float64)
    if precision == 1 and order % 2:          # the tensor cores take even orders only
        with pytest.raises(pb.AfmpbError, match="fmm_order"):
            pb.Handle.for_molecule(mol, order=order, leaf_cap=leaf_cap, precision=precision)
        return
    with pb.Handle.for_molecule(mol, order=order, leaf_cap=leaf_cap, precision=precision) as h:
        assert h.info()["n_m2l_pairs"] > 0
        y = far_parts(h, x)
        ref, _ = pair_sums(mol, o, whole_matrix(h), x)
    bar = order ** 2 * (3 + np.sqrt(8)) ** (1 - order) + 1e-4
    for block in (slice(None, mol.n_nodes), slice(mol.n_nodes, None)):
        err = np.linalg.norm(y[block] - ref[block]) / np.linalg.norm(ref[block])
        assert err < bar, (err, bar)
