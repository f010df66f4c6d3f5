"""The tensor-core M2L on levels blocked by octant (768 boxes and more) and on smaller ones,
with full, part-filled and last blocks: the same tree's product with the FP32 translations."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("subdiv,leaf_cap,order", [(3, 2, 6), (4, 2, 6), (4, 5, 6), (4, 5, 8), (5, 9, 6)])
def test_blocked_levels_match_fp32_translations(subdiv, leaf_cap, order):
    """The BF16 split keeps 16 bits of each factor (2^-16 = 1.5e-5 a product, three products);
    the bar is the product's 1e-4."""
    import torch
    import paper_1710_06316_gb300 as pb
    mol = synthetic.born_ion(subdiv=subdiv, radius=8.0)
    rng = np.random.default_rng(leaf_cap)
    mol.xyz = mol.xyz * (1 + 0.01 * rng.standard_normal((mol.n_nodes, 1)))
    x = torch.tensor(synthetic.random_unknowns(mol.n_nodes, subdiv).astype(np.float32), device="cuda")
    y = []
    for precision in (0, 1):
        with pb.Handle.for_molecule(mol, order=order, leaf_cap=leaf_cap, precision=precision) as h:
            level = np.bincount(h.tree()["level"])
            assert 0 < h.info()["m2l_rank"] <= 112       # the kernel in question
            out = torch.empty_like(x)
            h.matvec_parts(x, out, 2)
            h.sync()
            y.append(out.cpu().numpy().astype(np.float64))
    assert (level.max() >= 768) == (subdiv > 3)
    n = mol.n_nodes
    for block in (slice(None, n), slice(n, None)):
        assert np.linalg.norm(y[1][block] - y[0][block]) <= 1e-4 * np.linalg.norm(y[0][block])
