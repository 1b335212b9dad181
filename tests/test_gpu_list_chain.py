"""List chains (GOCP_ONCHIP_CHAINS=list, the default form from 15 qubits
complex64 / 12 qubits complex128 for problems built from integrals): forward
states, E and dE/dtheta against the oracle, the forward state bit for bit the
one of a launch per step, in one cluster and over every SM, with shares that
outgrow shared memory, a list that is given up for the enumerated pairs,
operators out of range, and a barrier wait that runs out.

Tolerances are those of tests/test_gpu_parity.py.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2607_15906_gb300 as gb  # noqa: E402
from oracle import mapping, pool as opool, statevector as sv  # noqa: E402
from oracle.pauli import PauliTable, parity  # noqa: E402
from synth import draw_ansatz, molecular_integrals  # noqa: E402

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = {"c128": (1e-10, 1e-10, 1e-10), "c64": (2e-5, 1e-6, 2e-6)}


def _host(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy().astype(np.complex128).ravel()


def _check(p, h, tabs, ref, ops, th, prec):
    n = p.n_qubits
    want = sv.prepare_state(sv.basis_state(n, ref), tabs, ops, th)
    d = p.new_states(1)[0]
    p.prepare_state(ops, th, d)
    assert np.max(np.abs(_host(d) - want)) <= TOL[prec][0] * np.max(np.abs(want))
    e, de = p.energy_grad(ops, th)
    e_ref, de_ref = sv.energy_grad(h, sv.basis_state(n, ref), tabs, ops, th)
    assert abs(e - e_ref) <= TOL[prec][1] * max(1.0, abs(e_ref))
    assert np.max(np.abs(de - de_ref)) <= TOL[prec][2] * max(1.0, np.max(np.abs(de_ref)))
    assert p.device_errors() == 0
    e2, de2 = p.energy_grad(ops, th)
    assert e2 == e and np.array_equal(de2, de)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb,n_elec,mp", [(4, 4, "jw"), (5, 3, "bk"), (6, 6, "jw"), (7, 6, "bk")])
def test_list_chain_matches_oracle(prec, n_orb, n_elec, mp, monkeypatch):
    """70 operators: more than one staged chunk of steps."""
    monkeypatch.setenv("GOCP_ONCHIP_CHAINS", "list")
    ints = molecular_integrals(n_orb, seed=n_orb, decay=True)
    h = mapping.hamiltonian_table(ints, mp)
    tabs = opool.pool_tables(2 * n_orb, n_elec, mp)
    p = gb.Problem.build(ints, n_elec, mapping=mp, precision=prec, device=0)
    ops, th = draw_ansatz(len(tabs), 70, seed=n_orb, theta_sigma=0.3)
    _check(p, h, tabs, p.info["ref_index"], ops, th, prec)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n", [8, 9])
def test_list_chain_given_up(prec, n, monkeypatch):
    """Generators with one-qubit x masks fill the state: the backward list
    passes a quarter of it and the sweep enumerates pairs."""
    monkeypatch.setenv("GOCP_ONCHIP_CHAINS", "list")
    rng = np.random.default_rng(70 + n)
    x = rng.integers(0, 1 << n, size=30)
    z = rng.integers(0, 1 << n, size=30)
    H = PauliTable(n, x, z, parity(x & z), rng.normal(size=30))
    gens = [PauliTable(n, np.array([1 << q]), np.array([1 << q]), np.array([0]), np.array([0.5])) for q in range(n)]
    to_t = lambda t: (t.x.astype(np.uint32), t.z.astype(np.uint32), (t.phase % 4).astype(np.uint8), t.coeff)
    p = gb.Problem.from_tables(n, to_t(H), [to_t(g) for g in gens], ref_index=0, precision=prec, device=0)
    ops = np.concatenate([np.arange(n), rng.integers(0, n, size=5)]).astype(np.int32)
    th = rng.uniform(0.2, 0.7, size=len(ops))
    _check(p, H, gens, 0, ops, th, prec)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb,share", [(7, None), (8, "64"), (9, None), (9, "64")])
def test_list_chain_equals_a_launch_per_step(prec, n_orb, share, monkeypatch):
    """Cluster and cooperative forms; share 64: entries beyond the first 64 of
    a block are read in place."""
    ints = molecular_integrals(n_orb, seed=1, decay=True)
    p = gb.Problem.build(ints, 8, precision=prec, int_drop=1e-3, device=0)
    ops, th = draw_ansatz(p.pool_size, 50, seed=3, theta_sigma=0.3)
    out = {}
    for mode in ("off", "list"):
        monkeypatch.setenv("GOCP_ONCHIP_CHAINS", mode)
        if share and mode == "list":
            monkeypatch.setenv("GOCP_LIST_SHARE", share)
        d = p.new_states(1)[0]
        p.prepare_state(ops, th, d)
        out[mode] = (d, *p.energy_grad(ops, th))
    assert p.device_errors() == 0
    assert torch.equal(out["off"][0], out["list"][0])
    assert out["off"][1] == out["list"][1]
    assert np.max(np.abs(out["off"][2] - out["list"][2])) <= TOL[prec][2] * max(1.0, np.max(np.abs(out["off"][2])))


def test_list_chain_flags_operators_out_of_range(monkeypatch):
    monkeypatch.setenv("GOCP_ONCHIP_CHAINS", "list")
    p = gb.Problem.build(molecular_integrals(8, seed=1, decay=True), 8, precision="c64", device=0)
    ops, th = draw_ansatz(p.pool_size, 6, seed=3)
    good = p.new_states(1)[0]
    p.prepare_state(np.delete(ops, 2), np.delete(th, 2), good)
    assert p.device_errors() == 0
    ops[2] = p.pool_size
    bad = p.new_states(1)[0]
    p.prepare_state(torch.from_numpy(ops).cuda(), torch.from_numpy(th).cuda(), bad)
    assert p.device_errors() == 1
    assert torch.equal(good, bad)      # the step acts as the identity


def test_list_chain_wait_runs_out(monkeypatch):
    """A zero limit makes every barrier wait give up at once: the call returns,
    the flag is reported, and the next call is correct again."""
    p = gb.Problem.build(molecular_integrals(9, seed=1, decay=True), 8, precision="c128", device=0)
    ops, th = draw_ansatz(p.pool_size, 12, seed=3)
    want = p.new_states(1)[0]
    p.prepare_state(ops, th, want)
    assert p.device_errors() == 0
    monkeypatch.setenv("GOCP_CHAIN_WAIT_NS", "0")
    got = p.new_states(1)[0]
    p.prepare_state(ops, th, got)
    assert p.device_errors() == 4
    monkeypatch.delenv("GOCP_CHAIN_WAIT_NS")
    p.prepare_state(ops, th, got)
    assert p.device_errors() == 0 and torch.equal(want, got)


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n_orb,n_elec", [(4, 3), (6, 6), (9, 8)])
def test_sector_chain_equals_a_launch_per_step(prec, n_orb, n_elec, monkeypatch):
    """The sector layout's chains in one launch (one block, and several waiting
    for one another; 70 operators: more than one staged chunk) against a launch
    per step: the state bit for bit, dE/dtheta to rounding, twice the same; an
    operator out of range is flagged and acts as the identity."""
    ints = molecular_integrals(n_orb, seed=2, decay=True)
    p = gb.Problem.build(ints, n_elec, precision=prec, device=0, sector=True)
    ops, th = draw_ansatz(p.pool_size, 70, seed=4, theta_sigma=0.3)
    out = {}
    for mode in ("off", None):
        if mode:
            monkeypatch.setenv("GOCP_ONCHIP_CHAINS", mode)
        else:
            monkeypatch.delenv("GOCP_ONCHIP_CHAINS")
        d = p.new_states(1)[0]
        p.prepare_state(ops, th, d)
        out[mode] = (d, *p.energy_grad(ops, th))
    assert p.device_errors() == 0
    assert torch.equal(out["off"][0], out[None][0]) and out["off"][1] == out[None][1]
    assert np.max(np.abs(out["off"][2] - out[None][2])) <= TOL[prec][2] * max(1.0, np.max(np.abs(out["off"][2])))
    e, de = p.energy_grad(ops, th)
    assert e == out[None][1] and np.array_equal(de, out[None][2])
    good, bad = p.new_states(2)
    p.prepare_state(np.delete(ops, 40), np.delete(th, 40), good)
    ops[40] = p.pool_size
    p.prepare_state(torch.from_numpy(ops).cuda(), torch.from_numpy(th).cuda(), bad)
    assert p.device_errors() == 1 and torch.equal(good, bad)
