"""The tile tuner's P2P parameter: the size of the work units.  The blocks resident per SM follow
from the kernel, so they are reported and not searched."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,order,subdiv", [(0, 4, 3), (0, 5, 4), (1, 4, 5), (1, 8, 4)])
def test_one_parameter_for_the_unit_size(precision, order, subdiv):
    import paper_1710_06316_gb300 as pb
    mol = synthetic.kirkwood_sphere(subdiv=subdiv)
    with pb.Handle.for_molecule(mol, order=order, precision=precision, leaf_cap=pb.LEAF_CAP_AUTO) as h:
        rep = h.autotune()
    assert rep["p2p_resident"] == 6 and rep["p2p_units_per_block"] in (1, 2, 3, 4, 6)
    assert 0 < rep["p2p_ms_tuned"] <= rep["p2p_ms_default"]
