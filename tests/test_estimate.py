"""The memory estimate that the server reserves by stays above what a solve holds at its peak, at
orders whose tables are small beside fixed-size parts (full-form tensor-core tiles, charge FMM)."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,order,leaf_cap,charge_fmm", [
    (0, 2, 0, 2), (0, 3, 0, 2), (0, 4, 64, 2), (0, 6, 0, 2), (1, 2, 0, 1), (1, 2, 16, 1), (1, 2, 64, 2), (1, 4, 0, 2),
    (1, 4, 4, 1), (1, 4, 64, 2), (1, 6, 0, 1), (1, 6, 0, 2)])
def test_estimate_is_above_the_peak(precision, order, leaf_cap, charge_fmm):
    import paper_1710_06316_gb300 as pb
    mol = synthetic.kirkwood_sphere(subdiv=6)
    options = dict(order=order, precision=precision, leaf_cap=leaf_cap, charge_fmm=charge_fmm)
    with pb.Handle.for_molecule(mol, **options) as h:
        h.solve(raise_on_noconv=False)
        h.energy()
        info = h.info()
    used = max(info["device_bytes"], info["device_bytes_peak"])
    estimate = pb.estimate_bytes(mol.n_nodes, len(mol.q), **options)
    assert used <= estimate, used / estimate


def test_estimate_of_uncompressed_tensor_core_translations():
    import paper_1710_06316_gb300 as pb
    mol = synthetic.kirkwood_sphere(subdiv=6)
    with pb.Handle.for_molecule(mol, order=6, precision=1, m2l_tol=-1.0) as h:
        h.solve(raise_on_noconv=False)
        info = h.info()
    used = max(info["device_bytes"], info["device_bytes_peak"])
    estimate = pb.estimate_bytes(mol.n_nodes, len(mol.q), order=6, precision=1, m2l_tol=-1.0)
    assert used <= estimate, used / estimate
