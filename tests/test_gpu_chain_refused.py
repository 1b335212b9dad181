"""Chains whose one launch is refused (GOCP_CHAIN_REFUSE=1 stands for the
driver's answer) take a launch per step: the same state and E bit for bit,
dE/dtheta to rounding (the bounds of tests/test_gpu_parity.py)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from synth import draw_ansatz, molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("sector", [False, True])
@pytest.mark.parametrize("n_orb", [8, 9])       # 9: the cooperative form in both precisions
def test_refused_launch_takes_a_launch_per_step(prec, sector, n_orb, monkeypatch):
    p = gb.Problem.build(molecular_integrals(n_orb, seed=1, decay=True), 8, precision=prec, int_drop=1e-3, device=0,
                         sector=sector)
    ops, th = draw_ansatz(p.pool_size, 40, seed=3, theta_sigma=0.3)
    out = []
    for refuse in ("0", "1"):
        monkeypatch.setenv("GOCP_CHAIN_REFUSE", refuse)
        d = p.new_states(1)[0]
        n0 = gb.launch_count()
        p.prepare_state(ops, th, d)
        e, de = p.energy_grad(ops, th)
        out.append((d, e, de, gb.launch_count() - n0))
    assert p.device_errors() == 0
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    assert np.max(np.abs(out[0][2] - out[1][2])) <= (1e-10 if prec == "c128" else 2e-6) * max(1.0, np.max(np.abs(out[0][2])))
    assert out[0][3] < 40 < out[1][3]
