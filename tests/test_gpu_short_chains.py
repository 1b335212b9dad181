"""Short forward chains (up to 24 operators of a problem built from integrals take
one cluster, more of them every SM): the state bit for bit that of a launch per
step at the lengths where the form changes, with operators that spread over many
determinants."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from synth import molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb", [8, 10])
@pytest.mark.parametrize("n_ops", [2, 13, 14, 24, 25])
def test_short_chain(prec, n_orb, n_ops, monkeypatch):
    p = gb.Problem.build(molecular_integrals(n_orb, seed=5, decay=True), n_orb, precision=prec, int_drop=1e-3, device=0)
    rng = np.random.default_rng(n_ops)
    # singles out of different orbitals first: each multiplies the amplitudes
    ops = np.concatenate([rng.integers(0, min(p.pool_size, 3 * n_orb), size=n_ops // 2),
                          rng.integers(0, p.pool_size, size=n_ops - n_ops // 2)]).astype(np.int32)
    th = rng.normal(0.0, 0.4, size=n_ops)
    out = {}
    for mode in ("off", None):
        if mode:
            monkeypatch.setenv("GOCP_ONCHIP_CHAINS", mode)
        else:
            monkeypatch.delenv("GOCP_ONCHIP_CHAINS")
        out[mode] = p.new_states(1)[0]
        p.prepare_state(ops, th, out[mode])
    assert torch.equal(out["off"], out[None]) and p.device_errors() == 0
