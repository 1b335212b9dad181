"""Scatter H psi with one block per tile (20 qubits and up) on random tables: the
group forms of test_gpu_scatter_cases.py with states of a few amplitudes (most
tiles have no live source and are written as zeros at once) and of many (units of
several chunks), and a table whose heads do not fit in shared memory.

Tolerances are those of tests/test_gpu_parity.py: 1e-10 (complex128) and 2e-5
(complex64) of the largest entry of H psi, 1e-10 and 1e-6 of max(1, |E|)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from oracle import statevector as sv  # noqa: E402
from oracle.pauli import PauliTable  # noqa: E402
from test_gpu_scatter_cases import TOL, _table  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _problem(H, prec):
    return gb.Problem.from_tables(H.n, (H.x.astype(np.uint32), H.z.astype(np.uint32), H.phase.astype(np.uint8), H.coeff),
                                  [], ref_index=0, precision=prec, device=0)


def _state(n, count, cplx, prec, rng):
    at = np.sort(rng.choice(1 << n, size=count, replace=False))
    v = rng.normal(size=count) + (1j * rng.normal(size=count) if cplx else 0.0)
    v = (v / np.linalg.norm(v)).astype(np.complex64 if prec == "c64" else np.complex128)
    d = torch.zeros(1 << n, dtype=torch.complex64 if prec == "c64" else torch.complex128, device="cuda:0")
    d[torch.from_numpy(at).cuda()] = torch.from_numpy(v).cuda()
    return at, v.astype(np.complex128), d


def _against_sparse(H, prec, at, v, d):
    """Every entry of H psi and E, from the terms times the few amplitudes."""
    p = _problem(H, prec)
    hd = torch.full_like(d, 7.0)
    e, nrm = p.energy(d, hd)
    ri, rv = sv.apply_terms_sparse(H, at, v)
    big = np.max(np.abs(rv))
    idx = torch.from_numpy(ri).cuda()
    err = hd[idx].cpu().numpy().astype(np.complex128) - rv
    assert np.max(np.abs(err)) <= TOL[prec][0] * big
    hd[idx] = 0.0
    assert int(torch.count_nonzero(hd)) == 0
    n2 = np.vdot(v, v).real
    e_ref = sv.sparse_dot(at, v, ri, rv).real / n2
    assert abs(e - e_ref) <= TOL[prec][1] * max(1.0, abs(e_ref)) and abs(nrm - n2) <= 1e-12
    p.close()


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n", [20, 21])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("count", [1, 5])
def test_few_amplitudes(prec, n, cplx, count):
    rng = np.random.default_rng(2000 + n)
    _against_sparse(_table(n, rng), prec, *_state(n, count, cplx, prec, rng))


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n", [20, 21])
@pytest.mark.parametrize("cplx", [False, True])
def test_many_amplitudes(prec, n, cplx, monkeypatch):
    """A ninth of the amplitudes: H psi at sampled rows, E from H psi."""
    monkeypatch.setenv("GOCP_SPARSE_FRAC", "0.25")
    rng = np.random.default_rng(3000 + n)
    H = _table(n, rng)
    at, v, d = _state(n, (1 << n) // 9 + 3, cplx, prec, rng)
    p = _problem(H, prec)
    hd = torch.empty_like(d)
    e, nrm = p.energy(d, hd)
    psi = d.cpu().numpy().astype(np.complex128)
    got = hd.cpu().numpy().astype(np.complex128)
    rows = np.concatenate([rng.integers(0, 1 << n, size=1500), at[:500], [0, (1 << n) - 1]])
    ref = sv.apply_terms_at(H, psi, rows)
    assert np.max(np.abs(got[rows] - ref)) <= TOL[prec][0] * np.max(np.abs(ref))
    n2 = np.vdot(psi, psi).real
    e_ref = np.vdot(psi, got).real / n2
    assert abs(e - e_ref) <= TOL[prec][1] * max(1.0, abs(e_ref)) and abs(nrm - n2) <= 1e-12
    p.close()


@pytest.mark.parametrize("prec", ["c128", "c64"])
def test_heads_beyond_shared_memory(prec):
    """26 qubits, 6,500 masks with as many patterns above the tile: a head of
    cases and a piece each, 104 KB of tile words."""
    n, rng = 26, np.random.default_rng(26)
    x = (rng.permutation(1 << 13)[:6500].astype(np.int64) << 13) | rng.integers(0, 1 << 13, size=6500)
    x = np.concatenate([x[x != 0], [0, 0]])
    z = np.concatenate([rng.integers(0, 1 << n, size=x.size - 1), [0]])
    H = PauliTable(n, x, z, np.zeros(x.size, np.int64), rng.normal(size=x.size))
    _against_sparse(H, prec, *_state(n, 300, True, prec, rng))
