"""The framework's work as its users have it done, case by case.

A case is one call of the public interface on seeded synthetic inputs (the
integral and angle distributions of synth/):

  eval    Problem.energy_grad: E and dE/dtheta of an ansatz, one evaluation of
          the re-optimisation (the call ADAPT makes most often)
  grad    ansatz_energy (torch.autograd) forward and backward: the same
          through an optimiser written in PyTorch
  select  Problem.adapt_step: the prepared state, H psi, E, every pool
          gradient and the selected operator, one per ADAPT iteration
  energy  Problem.energy on a state the caller brings: dense random
          amplitudes, for a molecular Hamiltonian or (spins) for one given as
          Pauli tables, which also reaches odd qubit counts
  serve   Server.submit / result: a burst of mixed-size energy+gradient
          requests, all queued at once

`exact` computes the same quantities in 64 bits from the definitions, in
second quantisation (ladder operators on occupation strings) or term by term
for Pauli tables, with torch alone.

E and the gradients of a complex64 problem come in float64 containers but are
single-precision results (FP32 amplitudes); they are returned as float32.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_15906_gb300 as gb
from paper_2607_15906_gb300.autograd import ansatz_energy
from paper_2607_15906_gb300.serving import Server

DEV = "cuda:0"
SIGMA = 0.05          # ansatz angles N(0, 0.05)


# ------------------------------------------------------------------ the cases

def _chem(name, kind, n_orb, n_elec, precision, **more):
    c = dict(name=name, kind=kind, n_orb=n_orb, n_elec=n_elec, precision=precision, mapping="jw",
             layout="full", n_ops=0, int_drop=0.0, host=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest problem (2 orbitals): what a call costs at all, with
        # host arrays as SciPy's BFGS hands them over
        _chem("eval_4q_c128", "eval", 2, 2, "c128", n_ops=5, host=True),
        # ADAPT to 30 operators at 14 qubits in complex128 under Bravyi-Kitaev:
        # the last re-optimisations, again from SciPy
        _chem("eval_14q_c128_bk", "eval", 7, 6, "c128", mapping="bk", n_ops=30, host=True),
        # a 60-parameter ansatz at 20 qubits differentiated by torch.autograd
        _chem("grad_20q_c64", "grad", 10, 10, "c64", n_ops=60),
        # the 24-qubit workload: a selection step on 100 operators, then an
        # evaluation of the grown ansatz, everything resident on the device
        _chem("select_24q_c64", "select", 12, 8, "c64", n_ops=100, int_drop=1e-3),
        _chem("eval_24q_c64", "eval", 12, 8, "c64", n_ops=101, int_drop=1e-3),
        # the same selection in double precision
        _chem("select_24q_c128", "select", 12, 8, "c128", n_ops=100, int_drop=1e-3),
        # the largest full layout of the benchmark that leaves room for three: 28 qubits, 2 GiB states
        _chem("select_28q_c64", "select", 14, 8, "c64", n_ops=100, int_drop=1e-3),
        # the sector layout of the 24-qubit workload
        _chem("eval_sector_24q_c64", "eval", 12, 8, "c64", n_ops=101, int_drop=1e-3, layout="sector"),
        # H psi and E of states that are not confined to a sector
        _chem("energy_dense_22q_c64", "energy", 11, 10, "c64"),
        _chem("energy_dense_18q_c128", "energy", 9, 8, "c128"),
        # a spin Hamiltonian given as Pauli tables, odd qubit count
        dict(name="energy_spins_19q_c64", kind="spins", n=19, precision="c64"),
        # serving: 28 requests of 10 to 22 qubits, 10 to 80 operators, queued together
        dict(name="serve_28_c64", kind="serve", requests=28, n_min=10, n_max=22, precision="c64"),
    ]


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "grad", "select", "select", "energy", "spins", "serve"])
    prec = rng.choice(["c64", "c64", "c128"])
    if kind == "spins":
        return dict(kind=kind, n=rng.randint(5, 21 if prec == "c64" else 18), precision=prec)
    if kind == "serve":
        lo = rng.choice([4, 6, 8, 10])
        return dict(kind=kind, requests=rng.randint(3, 28), n_min=lo, n_max=rng.choice([12, 14, 16, 18, 20, 22]),
                    precision="c64")
    if kind == "energy":
        n_orb = rng.randint(3, 11 if prec == "c64" else 9)
        return _draw_chem(rng, kind, n_orb, rng.randint(2, n_orb), prec, 0)
    while True:
        n_orb = rng.randint(2, 14 if prec == "c64" else 12)
        n_elec = rng.randint(2, min(10, 2 * n_orb - 2))
        if _dim(n_orb, n_elec) <= 260_000 or (n_orb == 14 and n_elec <= 8):
            break
    n_ops = int(round(math.exp(rng.uniform(math.log(3.0), math.log(110.0)))))
    return _draw_chem(rng, kind, n_orb, n_elec, prec, n_ops)


def _draw_chem(rng, kind, n_orb, n_elec, prec, n_ops):
    c = _chem("", kind, n_orb, n_elec, prec, n_ops=n_ops, mapping=rng.choice(["jw", "jw", "bk"]),
              int_drop=rng.choice([0.0, 1e-3]) if n_orb <= 10 else 1e-3,
              layout=rng.choice(["full", "full", "sector"]) if kind in ("eval", "select") else "full",
              host=kind in ("eval", "select") and rng.random() < 0.5)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _integrals(n_orb, seed):
    from synth import molecular_integrals
    return molecular_integrals(n_orb, seed=seed, decay=True)


def _pool_size(n_orb, n_elec):
    return len(_excitations(2 * n_orb, n_elec))


def _excitations(n, n_elec):
    """(occupied, virtual) spin-orbitals of the singles, then the doubles."""
    occ, vir = range(n_elec), range(n_elec, n)
    out = [((i,), (a,)) for i in occ for a in vir if (i - a) % 2 == 0]
    for i in occ:
        for j in range(i + 1, n_elec):
            for a in vir:
                for b in range(a + 1, n):
                    if i % 2 + j % 2 == a % 2 + b % 2:
                        out.append(((i, j), (a, b)))
    return out


def _ansatz(n_orb, n_elec, n_ops, seed):
    m = _pool_size(n_orb, n_elec)
    rng = np.random.default_rng([seed, 1])
    return (rng.integers(0, max(m, 1), size=n_ops).astype(np.int32), rng.normal(0.0, SIGMA, size=n_ops))


def _random_state(n, precision, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    dt = torch.float32 if precision == "c64" else torch.float64
    v = torch.randn((1 << n, 2), generator=g, device=DEV, dtype=dt)
    v /= torch.linalg.vector_norm(v)
    return torch.view_as_complex(v)


def _spin_terms(n, seed):
    """All-pairs Heisenberg couplings with random strengths, random X and Z
    fields: (x, z, phase, coeff), a term being coeff i^phase X^x Z^z with Z
    acting first (Y = i X Z)."""
    rng = np.random.default_rng([seed, 2])
    t = []
    for i in range(n):
        for j in range(i + 1, n):
            m, (a, b, c) = (1 << i) | (1 << j), rng.normal(0.0, 1.0 / math.sqrt(n), size=3)
            t += [(m, 0, 0, a), (m, m, 2, b), (0, m, 0, c)]
        t += [(1 << i, 0, 0, rng.normal()), (0, 1 << i, 0, rng.normal())]
    return t


def _spin_tables(n, seed):
    t = _spin_terms(n, seed)
    # neighbour rotations (s+_i s-_j - h.c.) as the pool
    gens = [([(1 << i) | (2 << i)] * 2, [1 << i, 2 << i], [0, 0], [0.5, -0.5]) for i in range(n - 1)]
    return [list(c) for c in zip(*t)], gens


def _requests(case, seed):
    """(n_orb, n_elec, integral seed, ansatz) of each request: sizes in turn,
    10 to 80 operators (the same lengths for every seed)."""
    sizes = list(range(case["n_min"], max(case["n_max"], case["n_min"]) + 1, 2))
    lengths = np.random.default_rng(case["requests"]).integers(10, 81, size=case["requests"])
    rng = np.random.default_rng([seed, 3])
    out = []
    for i in range(case["requests"]):
        n = sizes[i % len(sizes)]
        o, e = n // 2, 2 * (n // 4)
        s = int(rng.integers(1 << 30))
        out.append((o, e, s, _ansatz(o, e, int(lengths[i]), s)))
    return out


def _build(case, seed):
    return gb.Problem.build(_integrals(case["n_orb"], seed), case["n_elec"], mapping=case["mapping"],
                            precision=case["precision"], int_drop=case["int_drop"], device=0,
                            sector=case["layout"] == "sector")


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k, "single": case["precision"] == "c64"}
    if k == "serve":
        reqs = _requests(case, seed)
        s["server"] = Server(0, max_slots=128)
        s["requests"] = [(gb.Problem.build(_integrals(o, sd), e, precision=case["precision"], device=0),
                          ops, th) for o, e, sd, (ops, th) in reqs]
        return s
    if k == "spins":
        terms, gens = _spin_tables(case["n"], seed)
        p = gb.Problem.from_tables(case["n"], terms, gens, 1, precision=case["precision"], device=0)
    else:
        p = _build(case, seed)
    s["problem"] = p
    if k in ("spins", "energy"):
        s["psi"] = _random_state(p.n_qubits, case["precision"], seed)
        s["hpsi"] = torch.empty_like(s["psi"])
        s["e2"] = torch.zeros(2, dtype=torch.float64, device=DEV)
        return s
    ops, th = _ansatz(case["n_orb"], case["n_elec"], case["n_ops"], seed)
    s["ws"] = p.workspace()
    s["host"] = case["host"]
    if case["host"]:
        s["ops"], s["theta"] = ops, th
        return s
    s["ops"] = torch.from_numpy(ops).to(DEV) if k != "grad" else ops
    s["theta"] = torch.from_numpy(th).to(DEV)
    if k == "grad":
        s["theta"].requires_grad_(True)
    s["e2"] = torch.zeros(2, dtype=torch.float64, device=DEV)
    s["de"] = torch.zeros(max(len(ops), 1), dtype=torch.float64, device=DEV)
    s["grads"] = torch.zeros(max(p.pool_size, 1), dtype=torch.float64, device=DEV)
    s["sel"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    return s


def _out(s, v):
    """A result in the precision it was computed in."""
    if isinstance(v, torch.Tensor):
        return v.to(torch.float32) if s["single"] else v
    return np.asarray(v, dtype=np.float32 if s["single"] else np.float64)


def run(s):
    k = s["kind"]
    if k == "serve":
        tickets = [s["server"].submit(p, ops, th) for p, ops, th in s["requests"]]
        got = [s["server"].result(t) for t in tickets]
        return {"e": _out(s, np.array([e for e, _ in got])), "de": _out(s, np.concatenate([d for _, d in got]))}
    p = s["problem"]
    if k in ("spins", "energy"):
        p.energy(s["psi"], s["hpsi"], out=s["e2"])
        return {"hpsi": s["hpsi"], "e": _out(s, s["e2"])}
    if k == "grad":
        s["theta"].grad = None
        e = ansatz_energy(s["theta"], p, s["ops"], s["ws"])
        e.backward()
        return {"e": _out(s, e.detach()), "de": _out(s, s["theta"].grad)}
    if k == "eval":
        if s["host"]:
            e, de = p.energy_grad(s["ops"], s["theta"], ws=s["ws"])
            return {"e": _out(s, e), "de": _out(s, de)}
        p.energy_grad(s["ops"], s["theta"], ws=s["ws"], out_e=s["e2"], out_de=s["de"])
        return {"e": _out(s, s["e2"][:1]), "de": _out(s, s["de"])}
    if s["host"]:
        e, n2, g, sel = p.adapt_step(s["ops"], s["theta"], ws=s["ws"])
        return {"e": _out(s, np.array([e, n2])), "grads": _out(s, g), "selected": sel, "states": s["ws"]}
    p.adapt_step(s["ops"], s["theta"], ws=s["ws"], out=(s["e2"], s["grads"], s["sel"]))
    return {"e": _out(s, s["e2"]), "grads": _out(s, s["grads"]), "selected": s["sel"], "states": s["ws"]}


# ------------------------------------------------------------------ work

def _sector(n_orb, n_elec):
    return (n_elec + 1) // 2, n_elec // 2


def _dim(n_orb, n_elec):
    na, nb = _sector(n_orb, n_elec)
    return math.comb(n_orb, na) * math.comb(n_orb, nb)


def _connected(n_orb, na, nb):
    """Determinants that one determinant couples to through H."""
    va, vb = n_orb - na, n_orb - nb
    return (1 + na * va + nb * vb + math.comb(na, 2) * math.comb(va, 2) + math.comb(nb, 2) * math.comb(vb, 2) +
            na * va * nb * vb)


def _chem_flops(n_orb, n_elec, kind, n_ops):
    """H psi on the amplitudes the ansatz reaches (a real coupling times a
    complex amplitude, accumulated: 4), the Taylor steps on the pairs they
    touch (6 for the polynomial's 2 x 2 real matrix per component pair), the
    backward sweep (three times a step), the gradients (a complex product per
    touched amplitude)."""
    na, nb = _sector(n_orb, n_elec)
    d = _dim(n_orb, n_elec)
    nnz = d if n_ops > 40 else min(d, 1 << n_ops)
    touched = nnz * min(1.0, 2.0 * max(na, 1) * max(nb, 1) / max(n_orb * n_orb, 1))
    f = 4.0 * nnz * _connected(n_orb, na, nb) + 6.0 * n_ops * touched / 2
    if kind == "select":
        f += 4.0 * touched * _pool_size(n_orb, n_elec)
    else:
        f += 18.0 * n_ops * touched / 2
    return f


def work(case):
    k, amp = case["kind"], 8 if case["precision"] == "c64" else 16
    if k == "serve":
        reqs = _requests(case, 0)
        return {"bytes": float(sum(12 * len(a[0]) + 8 * len(a[0]) + 8 for _, _, _, a in reqs)),
                "flops": float(sum(_chem_flops(o, e, "eval", len(a[0])) for o, e, _, a in reqs))}
    if k == "spins":
        n = case["n"]
        return {"bytes": 2.0 * amp * 2 ** n, "flops": 4.0 * 2 ** n * (n * (n - 1) // 2 + n + 1)}
    if k == "energy":
        n_orb = case["n_orb"]
        # the mean number of couplings over all occupations of the n_orb orbitals
        w = [math.comb(n_orb, a) / 2.0 ** n_orb for a in range(n_orb + 1)]
        mean = sum(w[a] * w[b] * _connected(n_orb, a, b) for a in range(n_orb + 1) for b in range(n_orb + 1))
        return {"bytes": 2.0 * amp * 4 ** n_orb, "flops": 4.0 * 4 ** n_orb * mean}
    dim = _dim(case["n_orb"], case["n_elec"]) if case["layout"] == "sector" else 4 ** case["n_orb"]
    states = 2.0 * amp * dim if k == "select" else 0.0   # psi and H psi are results of a selection step
    return {"bytes": states + 12.0 * case["n_ops"] + 8.0 * case["n_ops"] + 8.0,
            "flops": float(_chem_flops(case["n_orb"], case["n_elec"], k, case["n_ops"]))}


# ------------------------------------------------------------------ exact values

def _parity(v):
    for s in (16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return v & 1


def _bk_rows(n):
    """Row j of the Fenwick-tree matrix: occupations j+1-lowbit(j+1) .. j."""
    rows = []
    for j in range(n):
        low = (j + 1) & -(j + 1)
        rows.append(sum(1 << i for i in range(j + 1 - low, j + 1)))
    return rows


class _Fock:
    """Determinants (occupation integers, ascending) and 64-bit vectors over
    them: tensors (D, c), c = 1 for real and 2 for complex amplitudes."""

    def __init__(self, n_orb, mapping, n_elec=None):
        self.n = 2 * n_orb
        if n_elec is None:
            self.keys = torch.arange(1 << self.n, device=DEV)
            self.all = True
        else:
            na, nb = _sector(n_orb, n_elec)
            spread = lambda c, s: [sum(1 << (2 * p + s) for p in range(n_orb) if (v >> p) & 1)
                                   for v in range(1 << n_orb) if bin(v).count("1") == c]
            a = torch.tensor(spread(na, 0), dtype=torch.int64, device=DEV)
            b = torch.tensor(spread(nb, 1), dtype=torch.int64, device=DEV)
            self.keys = (a[:, None] | b[None, :]).reshape(-1).sort().values
            self.all = False
        self.qubit = self.keys if mapping == "jw" else self._encode(self.keys)

    def _encode(self, keys):
        out = torch.zeros_like(keys)
        for j, row in enumerate(_bk_rows(self.n)):
            out |= _parity(keys & row) << j
        return out

    def at(self, occ):
        return occ if self.all else torch.searchsorted(self.keys, occ)

    def links(self, create, annihilate):
        """(to, from, sign) of the product of the creators (leftmost first)
        and annihilators (the last acts first) given, signs counting the
        occupied spin-orbitals below (Jordan-Wigner order)."""
        have = sum(1 << q for q in annihilate)
        free = sum(1 << p for p in create if not (have >> p) & 1)
        frm = torch.nonzero(((self.keys & have) == have) & ((self.keys & free) == 0)).reshape(-1)
        occ = self.keys[frm]
        odd = torch.zeros_like(occ)
        for q in reversed(annihilate):
            odd ^= _parity(occ & ((1 << q) - 1))
            occ = occ ^ (1 << q)
        for p in reversed(create):
            odd ^= _parity(occ & ((1 << p) - 1))
            occ = occ | (1 << p)
        return self.at(occ), frm, (1 - 2 * odd).to(torch.float64)[:, None]

    def hamiltonian(self, ints, drop, v):
        """H v: one- and two-body parts through E_pq = sum_s a+_ps a_qs,
        H = e0 + sum (h_pq - 1/2 sum_r (pr|rq)) E_pq + 1/2 sum (pq|rs) E_pq E_rs."""
        o = self.n // 2
        h = torch.tensor(np.where(np.abs(ints.h) < drop, 0.0, ints.h), device=DEV)
        g = torch.tensor(np.where(np.abs(ints.g) < drop, 0.0, ints.g), device=DEV)
        d, c = v.shape
        ev = torch.zeros((o * o, d * c), dtype=torch.float64, device=DEV)
        maps = {}
        for p in range(o):
            for q in range(o):
                row = ev[p * o + q].view(d, c)
                for s in (0, 1):
                    m = self.links((2 * p + s,), (2 * q + s,))
                    row.index_add_(0, m[0], m[2] * v[m[1]])
                    if d * o * o < 60_000_000:
                        maps[p, q, s] = m
        out = float(ints.e0) * v
        out += ((h - 0.5 * torch.einsum("prrq->pq", g)).reshape(1, -1) @ ev).view(d, c)
        step = max(1, 60_000_000 // (d * c))
        half = 0.5 * g.reshape(o * o, o * o)
        for r0 in range(0, o * o, step):
            w = half[r0:r0 + step] @ ev
            for i in range(w.shape[0]):
                p, q = divmod(r0 + i, o)
                for s in (0, 1):
                    m = maps.get((p, q, s)) or self.links((2 * p + s,), (2 * q + s,))
                    out.index_add_(0, m[0], m[2] * w[i].view(d, c)[m[1]])
        return out

    def generator(self, exc):
        """tau - tau^+ as the links of tau = a+_a a+_b a_j a_i (or a+_a a_i)."""
        occ, vir = exc
        return self.links(vir, tuple(reversed(occ)))

    @staticmethod
    def apply(gen, v):
        to, frm, sg = gen
        out = torch.zeros_like(v)
        out[to] = sg * v[frm]
        out[frm] -= sg * v[to]
        return out

    def taylor(self, gen, th, v, derivative=False):
        """sum_{m<=5} th^m / m! A^m v, or its derivative in th."""
        out = torch.zeros_like(v) if derivative else v.clone()
        w = v
        for m in range(1, 6):
            w = self.apply(gen, w)
            out += w * (th ** (m - 1) / math.factorial(m - 1) if derivative else th ** m / math.factorial(m))
        return out

    def full(self, v, n):
        """The amplitudes over the 2^n qubit basis states, complex."""
        out = torch.zeros(1 << n, dtype=torch.complex128, device=DEV)
        out[self.qubit] = torch.complex(v[:, 0], v[:, 1] if v.shape[1] == 2 else torch.zeros_like(v[:, 0]))
        return out

    def rows(self, v, n_orb, n_elec):
        """The amplitudes in the sector layout's row order: colexicographic
        rank of the alpha string, then of the beta string."""
        na, nb = _sector(n_orb, n_elec)
        strings = lambda c: torch.tensor([k for k in range(1 << n_orb) if bin(k).count("1") == c], device=DEV)
        spread = lambda k, s: sum((((k >> p) & 1) << (2 * p + s)) for p in range(n_orb))
        occ = (spread(strings(na), 0)[:, None] | spread(strings(nb), 1)[None, :]).reshape(-1)
        return torch.complex(v[self.at(occ), 0], torch.zeros_like(v[:, 0]))


def _prepared(n_orb, n_elec, mapping, ops, th, keep=False):
    f = _Fock(n_orb, mapping, n_elec)
    exc = _excitations(2 * n_orb, n_elec)
    v = torch.zeros((f.keys.numel(), 1), dtype=torch.float64, device=DEV)
    v[f.at(torch.tensor([(1 << n_elec) - 1], device=DEV))] = 1.0
    states, gens = [v], {}
    for k, t in zip(ops, th):
        if int(k) not in gens:
            gens[int(k)] = f.generator(exc[int(k)])
        v = f.taylor(gens[int(k)], float(t), v)
        if keep:
            states.append(v)
    return f, exc, v, states, gens


def _energy_grad(ints, n_orb, n_elec, mapping, drop, ops, th):
    f, _, v, states, gens = _prepared(n_orb, n_elec, mapping, ops, th, keep=True)
    hv = f.hamiltonian(ints, drop, v)
    n2 = float((v * v).sum())
    e = float((v * hv).sum()) / n2
    lam = (hv - e * v) / n2
    de = np.zeros(len(ops))
    for j in range(len(ops) - 1, -1, -1):
        g, t = gens[int(ops[j])], float(th[j])
        de[j] = 2.0 * float((lam * f.taylor(g, t, states[j], derivative=True)).sum())
        lam = f.taylor(g, -t, lam)   # A is antisymmetric: the transpose of T(t) is T(-t)
    return e, de


def exact(case, seed):
    k = case["kind"]
    if k == "serve":
        got = [_energy_grad(_integrals(o, s), o, e, "jw", 0.0, *a) for o, e, s, a in _requests(case, seed)]
        return {"e": np.array([x[0] for x in got]), "de": np.concatenate([x[1] for x in got])}
    if k == "spins":
        n = case["n"]
        psi = _random_state(n, case["precision"], seed).to(torch.complex128)
        b = torch.arange(1 << n, device=DEV)
        out = torch.zeros_like(psi)
        for x, z, ph, c in _spin_terms(n, seed):
            out += (c * 1j ** ph) * ((1 - 2 * _parity((b ^ x) & z)).to(torch.float64) * psi[b ^ x])
        n2 = float(torch.vdot(psi, psi).real)
        return {"hpsi": out, "e": np.array([float(torch.vdot(psi, out).real) / n2, n2])}
    ints = _integrals(case["n_orb"], seed)
    n, drop = 2 * case["n_orb"], case["int_drop"]
    if k == "energy":
        psi = _random_state(n, case["precision"], seed).to(torch.complex128)
        f = _Fock(case["n_orb"], case["mapping"])
        v = torch.view_as_real(psi[f.qubit])
        hv = f.hamiltonian(ints, drop, v)
        n2 = float((v * v).sum())
        return {"hpsi": f.full(hv, n), "e": np.array([float((v * hv).sum()) / n2, n2])}
    ops, th = _ansatz(case["n_orb"], case["n_elec"], case["n_ops"], seed)
    if k in ("eval", "grad"):
        e, de = _energy_grad(ints, case["n_orb"], case["n_elec"], case["mapping"], drop, ops, th)
        e = np.array([e]) if k == "eval" and not case["host"] else np.array(e)
        return {"e": e, "de": de}
    f, exc, v, _, _ = _prepared(case["n_orb"], case["n_elec"], case["mapping"], ops, th)
    hv = f.hamiltonian(ints, drop, v)
    n2 = float((v * v).sum())
    e = float((v * hv).sum()) / n2
    g = torch.empty(len(exc), dtype=torch.float64, device=DEV)
    for i, x in enumerate(exc):
        to, frm, sg = f.generator(x)
        g[i] = 2.0 * (sg * (hv[to] * v[frm] - hv[frm] * v[to])).sum() / n2
    if case["layout"] == "sector":
        states = torch.stack([f.rows(u, case["n_orb"], case["n_elec"]) for u in (v, hv)])
    else:
        states = torch.stack([f.full(u, n) for u in (v, hv)])
    return {"e": np.array([e, n2]), "grads": g, "selected": None, "states": states}
