"""The scatter H psi kernel's forms of a group against the oracle: LUT groups
of rank 0 to 3 split into cases (one, two, four or eight codes with one
magnitude, affine and other signs, all-different weights), term groups summed
through tables (with terms inside one index range, among the tile's bits, and
across ranges), a group that stays a list, the diagonal in several pieces, and
tiles smaller than, equal to and more than the kernel's 2^13 amplitudes.  Real
amplitudes (whose imaginary products are not formed) and complex ones.

Tolerances are those of tests/test_gpu_parity.py: 1e-10 (complex128) and 2e-5
(complex64) of the largest entry of H psi, 1e-10 and 1e-6 of max(1, |E|).
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from oracle import statevector as sv  # noqa: E402
from oracle.pauli import PauliTable, parity  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = {"c128": (1e-10, 1e-10), "c64": (2e-5, 1e-6)}


def _table(n, rng):
    x, z, c = [], [], []

    def group(gx, zs, ws):
        # weights as the kernel sees them at the output index: w = c (-1)^popc(x & z)
        for gz, w in zip(zs, ws):
            x.append(gx)
            z.append(int(gz))
            c.append(float(w) * (1 - 2 * int(parity(np.array([gx & int(gz)]))[0])))

    top = 1 << (n - 1)
    masks = rng.permutation(np.arange(1, 1 << n))[:40].tolist() + [1, 3, 1 << 12 if n > 12 else 1 << 11, top | 1, top]
    for i, gx in enumerate(dict.fromkeys(masks)):
        rank = i % 4
        v = [int(m) for m in rng.integers(1, 1 << n, size=rank)]
        zs = [int(rng.integers(0, 1 << n))]
        for m in v:
            zs += [q ^ m for q in zs]
        zs = list(dict.fromkeys(zs))
        kind = (i // 4) % 3
        ws = np.ones(len(zs)) / len(zs) if kind == 0 else rng.choice([-0.25, 0.25], size=len(zs)) if kind == 1 \
            else rng.normal(size=len(zs))
        group(gx, zs, ws)
    # around a centre: single bits over all ranges, and three masks across ranges
    for gx in (5 | top, 6):
        zc = int(rng.integers(0, 1 << n))
        ys = [0] + [1 << q for q in range(n)] + [(1 << 4) | (1 << 5), (1 << 8) | (1 << 9), 1 | top]
        zs = [zc ^ y for y in ys]
        group(gx, zs, rng.normal(size=len(zs)))
    # a list: random masks
    group(9, rng.permutation(1 << n)[:14], rng.normal(size=14))
    # the diagonal, more than one piece of 64 terms, and the identity
    dz = [0] + [1 << q for q in range(n)] + [(1 << q) | (1 << r) for q in range(n) for r in range(q)]
    group(0, dz, rng.normal(size=len(dz)))
    return PauliTable(n, np.array(x, np.int64), np.array(z, np.int64), np.zeros(len(x), np.int64), np.array(c))


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n", [12, 13, 14, 17])
@pytest.mark.parametrize("kind", ["real", "complex"])
def test_scatter_cases(prec, n, kind, monkeypatch):
    if prec == "c64" and n < 13:
        pytest.skip("complex64 takes the untiled kernel below 13 qubits")
    monkeypatch.setenv("GOCP_SPARSE_FRAC", "0.25")
    rng = np.random.default_rng(1000 + n)
    H = _table(n, rng)
    p = gb.Problem.from_tables(n, (H.x.astype(np.uint32), H.z.astype(np.uint32), H.phase.astype(np.uint8), H.coeff),
                               [], ref_index=0, precision=prec, device=0)
    psi = np.zeros(1 << n, np.complex128)
    at = rng.permutation(1 << n)[:(1 << n) // 9 + 3]      # ragged, below the quarter the list holds
    psi[at] = rng.normal(size=at.size) + (1j * rng.normal(size=at.size) if kind == "complex" else 0.0)
    psi /= np.linalg.norm(psi)
    d = torch.from_numpy(psi.astype(np.complex64 if prec == "c64" else np.complex128)).cuda()
    psi_in = d.cpu().numpy().astype(np.complex128)
    hd = torch.empty_like(d)
    e, nrm = p.energy(d, hd)
    ref = sv.apply_terms(H, psi_in)
    got = hd.cpu().numpy().astype(np.complex128)
    assert np.max(np.abs(got - ref)) <= TOL[prec][0] * np.max(np.abs(ref))
    e_ref = np.vdot(psi_in, ref).real / np.vdot(psi_in, psi_in).real
    assert abs(e - e_ref) <= TOL[prec][1] * max(1.0, abs(e_ref))
    assert abs(nrm - np.vdot(psi_in, psi_in).real) <= 1e-12
