"""GOCP_ONCHIP_CHAINS and the sector layout: unset and "list" run a chain in one
launch, the other values one launch per step; the state is the same bit for bit."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from synth import draw_ansatz, molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def test_forms(monkeypatch):
    p = gb.Problem.build(molecular_integrals(7, seed=1, decay=True), 6, precision="c64", device=0, sector=True)
    ops, th = draw_ansatz(p.pool_size, 30, seed=3)
    states = {}
    for mode, one in ((None, True), ("list", True), ("off", False), ("block", False), ("all", False)):
        if mode:
            monkeypatch.setenv("GOCP_ONCHIP_CHAINS", mode)
        d = p.new_states(1)[0]
        n0 = gb.launch_count()
        p.prepare_state(ops, th, d)
        assert (gb.launch_count() - n0 < 30) == one, mode
        states[mode] = d
    assert all(torch.equal(d, states[None]) for d in states.values())
