"""A chain's wait that runs out (GOCP_CHAIN_WAIT_NS=0) is returned by the calls
that read their results back: gocp_energy_grad and gocp_adapt_step with host
arrays.  The flag stays for gocp_device_errors, and the next call is correct."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from paper_2607_15906_gb300._lib import GOCP_ETIMEDOUT, GocpError  # noqa: E402
from synth import draw_ansatz, molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("sector", [False, True])
@pytest.mark.parametrize("call", ["energy_grad", "adapt_step"])
def test_host_calls_report_a_wait_that_ran_out(sector, call, monkeypatch):
    p = gb.Problem.build(molecular_integrals(9, seed=1, decay=True), 8, precision="c128", device=0, sector=sector)
    ops, th = draw_ansatz(p.pool_size, 12, seed=3)
    want = getattr(p, call)(ops, th)
    monkeypatch.setenv("GOCP_CHAIN_WAIT_NS", "0")
    with pytest.raises(GocpError) as info:
        getattr(p, call)(ops, th)
    assert info.value.code == GOCP_ETIMEDOUT
    monkeypatch.delenv("GOCP_CHAIN_WAIT_NS")
    got = getattr(p, call)(ops, th)       # the flag is still set; this call's own waits held
    assert p.device_errors() == 4 and p.device_errors() == 0
    for a, b in zip(want, got):
        assert np.allclose(a, b, rtol=0.0, atol=1e-10 * max(1.0, float(np.max(np.abs(a)))))
