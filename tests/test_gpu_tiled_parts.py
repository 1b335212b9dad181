"""Staged H psi with several blocks per tile where one piece holds most of the
groups: every block's part ends at its own last piece.  H psi and E of dense
states against the oracle, at the tolerances of tests/test_gpu_parity.py (1e-10
and, complex64, 2e-5 of the largest entry; 1e-10 and 1e-6 of max(1, |E|))."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from oracle import statevector as sv  # noqa: E402
from oracle.pauli import PauliTable, parity  # noqa: E402
from synth import random_state  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = {"c128": (1e-10, 1e-10), "c64": (2e-5, 1e-6)}


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n", [15, 16, 18])
@pytest.mark.parametrize("heavy", ["first", "middle", "own"])
def test_uneven_pieces(prec, n, heavy, monkeypatch):
    """41 masks of one pattern above the tile, single masks on up to five others;
    heavy "own": the pattern is zero, the tile's own (the last piece)."""
    monkeypatch.setenv("GOCP_SPARSE_FRAC", "0")
    lb = 13 if prec == "c64" else 12
    rng = np.random.default_rng(n)
    his = list(range(1, min(6, 1 << (n - lb))))
    pat = {"first": his[0], "middle": his[len(his) // 2], "own": 0}[heavy]
    x = [(pat << lb) | int(v) for v in rng.permutation(np.arange(1, 1 << lb))[:41]] + \
        [(h << lb) | int(rng.integers(0, 1 << lb)) for h in his]
    x = np.array(list(dict.fromkeys(x)) + [0], np.int64)
    z = rng.integers(0, 1 << n, size=x.size)
    H = PauliTable(n, x, z, parity(x & z), rng.normal(size=x.size))
    p = gb.Problem.from_tables(n, (x.astype(np.uint32), z.astype(np.uint32), (H.phase % 4).astype(np.uint8), H.coeff),
                               [], ref_index=0, precision=prec, device=0)
    psi = torch.from_numpy(random_state(n, seed=n).astype(np.complex64 if prec == "c64" else np.complex128)).cuda()
    hpsi = torch.empty_like(psi)
    e, _ = p.energy(psi, hpsi)
    assert p.device_errors() == 0
    v = psi.cpu().numpy().astype(np.complex128)
    ref = sv.apply_terms(H, v)
    got = hpsi.cpu().numpy().astype(np.complex128)
    assert np.max(np.abs(got - ref)) <= TOL[prec][0] * np.max(np.abs(ref))
    e_ref = np.vdot(v, ref).real / np.vdot(v, v).real
    assert abs(e - e_ref) <= TOL[prec][1] * max(1.0, abs(e_ref))
    p.close()
