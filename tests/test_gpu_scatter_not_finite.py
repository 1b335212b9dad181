"""H psi of a state with an amplitude that is not a number or infinite, on the
scatter kernel: the amplitude's own entry is not finite (its diagonal product
is not), and neither are E and <psi|psi>.  One and several blocks per tile."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from synth import draw_ansatz, molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb", [7, 10])
@pytest.mark.parametrize("value", [complex(float("nan"), 0.0), complex(0.5, float("nan")), complex(float("inf"), 0.0)])
def test_not_finite(prec, n_orb, value):
    p = gb.Problem.build(molecular_integrals(n_orb, seed=1, decay=True), 6, precision=prec, int_drop=1e-3, device=0)
    ops, th = draw_ansatz(p.pool_size, 12, seed=3)
    psi, hpsi = p.new_states(2)
    p.prepare_state(ops, th, psi)
    at = int(torch.nonzero(psi)[1])
    psi[at] = value
    e, nrm = p.energy(psi, hpsi)
    assert not np.isfinite(e) and not np.isfinite(nrm)
    assert not bool(torch.isfinite(torch.view_as_real(hpsi[at])).all())
    p.apply_h(psi, hpsi)
    assert not bool(torch.isfinite(torch.view_as_real(hpsi[at])).all())
    psi[at] = 0.25       # and none of it stays
    e, nrm = p.energy(psi, hpsi)
    assert np.isfinite(e) and bool(torch.isfinite(torch.view_as_real(hpsi)).all())
    assert p.device_errors() == 0
