"""Device memory of small problems: lists, inboxes and the sums of blocks that
share a tile are sized by the state, without a floor of megabytes."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from synth import molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n_orb,n_elec,prec", [(6, 6, "c128"), (7, 6, "c64"), (7, 6, "c128"), (8, 8, "c64")])
def test_device_bytes(n_orb, n_elec, prec):
    """At most 15 states of parts, one of split accumulators, four of lists and
    masks, and the tables (below four states at 12 to 16 qubits)."""
    p = gb.Problem.build(molecular_integrals(n_orb, seed=5, decay=True), n_elec, precision=prec, device=0)
    assert p.info["device_bytes"] <= 24 * p.state_bytes()
    p.close()
