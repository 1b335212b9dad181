"""List chains, call after call: the state and E of every call bit for bit those
of a launch per step, dE/dtheta the same to the rounding of its sum in every call
(the order of new entries is not fixed); and forward chains whose inboxes overflow
(GOCP_LIST_INBOX), which go over to the enumerated pairs."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from synth import draw_ansatz, molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _per_step(p, ops, th, monkeypatch):
    monkeypatch.setenv("GOCP_ONCHIP_CHAINS", "off")
    d = p.new_states(1)[0]
    p.prepare_state(ops, th, d)
    e, de = p.energy_grad(ops, th)
    return d, e, de


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb,n_elec,n_ops,repeats", [(7, 6, 65, 100), (9, 8, 33, 100), (9, 8, 65, 100),
                                                        (10, 10, 65, 50), (12, 8, 65, 20)])
def test_every_call_gives_the_same(prec, n_orb, n_elec, n_ops, repeats, monkeypatch):
    """33 and 65 operators: chains that stage descriptors between steps (every
    32nd), where blocks drift furthest apart."""
    p = gb.Problem.build(molecular_integrals(n_orb, seed=5, decay=True), n_elec, precision=prec, int_drop=1e-3, device=0)
    ops, th = draw_ansatz(p.pool_size, n_ops, seed=6, theta_sigma=0.3)
    want, e0, _ = _per_step(p, ops, th, monkeypatch)
    monkeypatch.setenv("GOCP_ONCHIP_CHAINS", "list")
    d = p.new_states(1)[0]
    ws = p.workspace()
    first = None
    # at most 1e5 terms of dE_j, summed in 53 bits (complex128) or 48 (complex64) in another order
    tol = 1e5 * (2.0 ** -53 if prec == "c128" else 2.0 ** -48)
    for _ in range(repeats):
        p.prepare_state(ops, th, d)
        assert torch.equal(d, want)
        e, de = p.energy_grad(ops, th, ws=ws)
        assert e == e0
        first = de if first is None else first
        assert np.max(np.abs(de - first)) <= tol * max(1.0, np.max(np.abs(first)))
    assert p.device_errors() == 0


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb,inbox", [(6, "1"), (7, "2"), (8, "5"), (9, "40")])
def test_forward_inbox_overflow(prec, n_orb, inbox, monkeypatch):
    p = gb.Problem.build(molecular_integrals(n_orb, seed=7, decay=True), 6, precision=prec, int_drop=1e-3, device=0)
    ops, th = draw_ansatz(p.pool_size, 50, seed=8, theta_sigma=0.3)
    want, e0, de0 = _per_step(p, ops, th, monkeypatch)
    monkeypatch.setenv("GOCP_ONCHIP_CHAINS", "list")
    monkeypatch.setenv("GOCP_LIST_INBOX", inbox)
    d = p.new_states(1)[0]
    for _ in range(20):
        p.prepare_state(ops, th, d)
        assert torch.equal(d, want)
    e, de = p.energy_grad(ops, th)
    assert e == e0
    # the bounds of tests/test_gpu_parity.py for dE/dtheta
    assert np.max(np.abs(de - de0)) <= (1e-10 if prec == "c128" else 2e-6) * max(1.0, np.max(np.abs(de0)))
    assert p.device_errors() == 0
