"""Scatter H psi, complex64: the weights of a term group far smaller than the
largest keep their precision.  Outputs that only the small group feeds are held
to the rounding that the kernel states: half a unit of the fixed-point scale 2^F
for the product, 2^-31 of the group's scale per term for the weight, and 2^-22 for
the FP32 weights and products."""

import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from oracle import statevector as sv  # noqa: E402
from oracle.pauli import PauliTable, parity  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _problem(n, groups, diagonal=()):
    """groups: (x, z masks, weights at the output index); diagonal: (z, weight)."""
    x, z, c = [], [], []
    for gx, zs, ws in groups:
        for gz, w in zip(zs, ws):
            x.append(gx)
            z.append(int(gz))
            c.append(float(np.float32(w)) * (1 - 2 * int(parity(np.array([gx & int(gz)]))[0])))
    for gz, w in diagonal:
        x.append(0)
        z.append(gz)
        c.append(float(w))
    H = PauliTable(n, np.array(x, np.int64), np.array(z, np.int64), np.zeros(len(x), np.int64), np.array(c))
    p = gb.Problem.from_tables(n, (H.x.astype(np.uint32), H.z.astype(np.uint32), H.phase.astype(np.uint8), H.coeff),
                               [], ref_index=0, precision="c64", device=0)
    return H, p


def _run(p, psi):
    d = torch.from_numpy(psi.astype(np.complex64)).cuda()
    hd = torch.empty_like(d)
    p.energy(d, hd)
    return hd.cpu().numpy().astype(np.complex128)


def _scale(hbound, dmax, m):
    """F of the call: sums below 2^62, off-diagonal products below 2^30."""
    return min(62 - math.frexp(2.0 * hbound * m)[1], 30 - math.frexp(2.0 * dmax * m)[1])


@pytest.mark.parametrize("n", [14, 17])
@pytest.mark.parametrize("small", [2.0 ** -8, 2.0 ** -14])
def test_small_term_group_keeps_its_weights(n, small, monkeypatch):
    monkeypatch.setenv("GOCP_SPARSE_FRAC", "0.25")
    rng = np.random.default_rng(n)
    groups = []
    for gx, size in ((5, 1.0), (6, small)):
        zc = int(rng.integers(0, 1 << n))
        zs = [zc ^ y for y in [0] + [1 << q for q in range(n)]]
        groups.append((gx, zs, size * rng.normal(size=len(zs))))
    H, p = _problem(n, groups)
    at = rng.permutation(1 << n)[:400]
    m = 0.05
    psi = np.zeros(1 << n, np.complex128)
    psi[at] = float(np.float32(m)) * rng.choice([-1.0, 1.0], size=at.size)
    got, ref = _run(p, psi), sv.apply_terms(H, psi)
    only = np.setdiff1d(at ^ 6, at ^ 5)
    sums = [float(np.sum(np.abs(w))) for _, _, w in groups]
    F = _scale(sum(sums), max(sums), m)
    tol = 2.0 ** -(F + 1) + m * sums[1] * (2.0 ** -22 + len(groups[1][1]) * 2.0 ** -30)
    assert np.max(np.abs(got[only] - ref[only])) <= tol


def test_large_constant_leaves_the_products_their_precision(monkeypatch):
    """A constant 2^30 times the largest off-diagonal weight: outputs without an
    amplitude of their own are held to half a unit of 2^F per product."""
    monkeypatch.setenv("GOCP_SPARSE_FRAC", "0.25")
    n, m = 15, 0.05
    rng = np.random.default_rng(3)
    groups = []
    for gx in (5, 6, 1 << (n - 1)):
        zc = int(rng.integers(0, 1 << n))
        zs = [zc ^ y for y in [0] + [1 << q for q in range(n)]]
        groups.append((gx, zs, rng.normal(size=len(zs))))
    groups.append((9, [3], [0.7]))          # a LUT group
    sums = [float(np.sum(np.abs(w))) for _, _, w in groups]
    H, p = _problem(n, groups, diagonal=[(0, 2.0 ** 30 * max(sums)), (7, 1.5)])
    at = rng.permutation(1 << n)[:400]
    psi = np.zeros(1 << n, np.complex128)
    psi[at] = float(np.float32(m)) * rng.choice([-1.0, 1.0], size=at.size)
    got, ref = _run(p, psi), sv.apply_terms(H, psi)
    off = np.setdiff1d(np.concatenate([at ^ g[0] for g in groups]), at)
    F = _scale(2.0 ** 30 * max(sums) + 1.5 + sum(sums), max(sums), m)
    tol = len(groups) * (2.0 ** -(F + 1) + m * max(sums) * (2.0 ** -22 + n * 2.0 ** -30))
    assert F == 30 - math.frexp(2.0 * max(sums) * m)[1]
    assert np.max(np.abs(got[off] - ref[off])) <= tol
    own = np.abs(got[at] - ref[at]) / np.abs(ref[at])
    assert np.max(own) <= 2.0 ** -22
