"""The work that a user of the simulator has it do, as timed cases.

Six kinds of pass, each through the public Python entry points:

  qsu     reset + apply_circuit: a circuit run whose state is the result
  energy  reset + apply_circuit + expect: one energy evaluation with every
          string's expectation value (a VQE without gradients, a readout)
  grad    autograd.vqe_energy + backward: one iteration of a VQE training
          loop (forward circuit, lambda = H psi, adjoint sweep)
  step    StateVector.vqe_step: the same iteration with the expectation value
          of every string besides (the benchmark's step)
  batch   batch_run: many small independent VQE states in one launch
  chunk   expect_noalloc: the strings of one tile on a caller-owned state, as
          each rank of a sharded state evaluates them on its chunk

Sizes are those of the repository's own workloads (workloads.CONFIGS) and of
their smaller copies: n = 12 to 30 qubits in complex64, 12 to 22 in
complex128.  Values that a complex64 state gives are kept in single precision
(the energy in one row with the values it belongs to), those of a complex128
state in double.

exact() is a plain gate-by-gate and string-by-string simulation in complex128
torch, in logical qubit order; it uses nothing of the simulator but the drawn
gate lists and strings.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_04252_gb300 import sv
from paper_2410_04252_gb300 import workloads as W
from paper_2410_04252_gb300.autograd import vqe_energy

SCHEDULES = {"lazy": sv.LAZY, "eager": sv.EAGER, "direct": sv.DIRECT}


def listed():
    return [
        # the smallest workload: complex128 under the ad hoc schedule; launches and host work
        dict(name="energy_hea_n12_c128_eager", kind="energy", n=12, g=2, dtype="c128", ansatz="hea", layers=4,
             ham="random", nterms=64, schedule="eager"),
        # a training iteration at the size that gradients are checked at (the n = 14 copy of the adjoint workload)
        dict(name="grad_hea_n14_c64", kind="grad", n=14, g=4, dtype="c64", ansatz="hea", layers=6,
             ham="random", nterms=1024, schedule="lazy"),
        # a chemistry-shaped training iteration at the size its error is stated at (the n = 20 copy)
        dict(name="grad_fabric_jw_n20_c64", kind="grad", n=20, g=4, dtype="c64", ansatz="fabric", layers=12,
             ham="jw", nterms=4096, schedule="lazy"),
        # a rank's chunk of a sharded state: one tile's strings, odd size, no allocation
        dict(name="chunk_random_n25_c64", kind="chunk", n=25, g=0, dtype="c64", ansatz="hea", layers=1,
             ham="random", nterms=96, schedule="lazy"),
        # dense 1-, 2- and 4-qubit matrices among rotations, odd size
        dict(name="qsu_mats_n23_c64", kind="qsu", n=23, g=5, dtype="c64", ansatz="mats", layers=120,
             ham="none", nterms=0, schedule="lazy"),
        # the state update of the particle-conserving ansatz, at its own size
        dict(name="qsu_fabric_n26_c64", kind="qsu", n=26, g=4, dtype="c64", ansatz="fabric", layers=8,
             ham="none", nterms=0, schedule="lazy"),
        # the chemistry-shaped energy with all 4096 strings (the n = 30 workload, two qubits fewer)
        dict(name="energy_fabric_jw_n28_c64", kind="energy", n=28, g=6, dtype="c64", ansatz="fabric", layers=12,
             ham="jw", nterms=4096, schedule="lazy"),
        # the adjoint workload's training iteration through autograd (odd size)
        dict(name="grad_hea_n27_c64", kind="grad", n=27, g=6, dtype="c64", ansatz="hea", layers=6,
             ham="random", nterms=1024, schedule="lazy"),
        # double precision, the paper's own: a whole step of the adjoint workload
        dict(name="step_hea_n22_c128", kind="step", n=22, g=4, dtype="c128", ansatz="hea", layers=6,
             ham="random", nterms=1024, schedule="lazy"),
        # the benchmark's step as large as a pass may be (the n = 32 workload, two qubits fewer)
        dict(name="step_hea_n30_c64", kind="step", n=30, g=6, dtype="c64", ansatz="hea", layers=6,
             ham="random", nterms=1024, schedule="lazy"),
        # the batched workload
        dict(name="batch256_hea_n18_c64", kind="batch", n=18, g=0, dtype="c64", ansatz="hea", layers=8, count=256,
             ham="random", nterms=512, schedule="lazy"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["qsu", "energy", "energy", "grad", "grad", "step", "batch", "chunk"])
    dtype = "c128" if rng.random() < 0.25 else "c64"
    c = dict(kind=kind, n=0, g=0, dtype=dtype, ansatz=rng.choice(["hea", "fabric"]), layers=0,
             ham=rng.choice(["random", "jw"]), nterms=_log_int(rng, 64, 1024), schedule="lazy")
    if kind == "batch":
        c.update(n=rng.randint(10, 18), ansatz="hea", layers=rng.randint(2, 8), count=_log_int(rng, 16, 256),
                 nterms=_log_int(rng, 64, 512))
        if dtype == "c128":
            c.update(n=min(c["n"], 13), nterms=min(c["nterms"], 256))
        return c
    top = {"qsu": 27, "energy": 27, "grad": 26, "step": 26, "chunk": 27}[kind] if dtype == "c64" else 22
    c["n"] = rng.randint(12, top)
    c["layers"] = rng.randint(3, 6) if c["ansatz"] == "hea" else rng.randint(6, 12)
    c["g"] = rng.randint(2, 6)
    if c["ansatz"] == "fabric":
        c["ham"] = "jw"            # random strings do not conserve the particle number: their values would be rounding
    if kind == "chunk":
        c.update(g=0, ansatz="hea", layers=1, nterms=_log_int(rng, 16, 256))
    if kind == "qsu":
        c.update(ham="none", nterms=0)
        if rng.random() < 0.3:
            c.update(ansatz="mats", layers=rng.randint(40, 160))
    if kind in ("energy", "grad", "step") and c["ham"] == "jw":
        c["nterms"] *= 4
    if c["n"] <= 20 and rng.random() < 0.2:
        c["schedule"] = rng.choice(["eager", "direct"])
    return c


# ------------------------------------------------------------------ inputs --

def _mats_circuit(n, m, seed):
    """A random gate list (the same for every seed) over every gate kind, the
    dense 1-, 2- and 4-qubit unitaries with matrices of their own."""
    rng = W.SplitMix64(17 + 100 * n + m)
    gates, mats, params, offset = [], [], 0, 0
    for i in range(m):
        kind = (W.RY, W.RZ, W.MAT1, W.CZ, W.MAT2, W.GIVENS, W.RY, W.MAT4)[rng.randint(8)]
        qs = []
        while len(qs) < W.GATE_NQ[kind]:
            q = rng.randint(n)
            if q not in qs:
                qs.append(q)
        p = mat = -1
        if kind in (W.RY, W.RZ, W.GIVENS):
            p, params = params, params + 1
        if kind in (W.MAT1, W.MAT2, W.MAT4):
            dim = 1 << W.GATE_NQ[kind]
            mats.append(W.random_unitary_mats(1, dim, (seed + 17) * 1000 + i))
            mat, offset = offset, offset + dim * dim
        gates.append((kind, tuple(qs), p, mat))
    return W._circuit(n, gates, params, np.concatenate(mats) if mats else None)


def _circuit(case, seed):
    n, layers = case["n"], case["layers"]
    if case["ansatz"] == "hea":
        return W.hea_circuit(n, layers)
    if case["ansatz"] == "fabric":
        return W.fabric_circuit(n, layers)
    return _mats_circuit(n, layers, seed)


def _hamiltonian(case, seed):
    make = W.jw_hamiltonian if case["ham"] == "jw" else W.random_hamiltonian
    return make(case["n"], case["nterms"], 2000 + seed) if case["nterms"] else None


def _params(case, count, seed):
    lo, hi = (0.0, 2.0 * math.pi) if case["ansatz"] == "hea" else (-math.pi, math.pi)
    p = W.uniform_params(count, 1000 + seed, lo, hi)
    # a single-precision program's parameters (autograd takes them as a float32 tensor)
    return p.astype(np.float32).astype(np.float64) if case["kind"] == "grad" and case["dtype"] == "c64" else p


def _init(case):
    return W.half_filled_index(case["n"]) if case["ansatz"] == "fabric" else 0


def _batch(case, seed):
    """(circuits, parameters) of the batched states: state i's depth, from 2
    up to the case's, is its own and stays; its parameters are drawn."""
    circs, params = [], []
    for i in range(case["count"]):
        circ = W.hea_circuit(case["n"], 2 + W.SplitMix64(3000 + i).randint(case["layers"] - 1))
        circs.append(circ)
        params.append(W.uniform_params(circ.nparams, 3000 + 1009 * (seed + 1) + i, 0.0, 2.0 * math.pi))
    return circs, params


def _chunk_state(case, seed):
    """A random state vector of norm 1 on the GPU (amplitudes of equal spread,
    as a deep circuit leaves them)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dt = torch.float32 if case["dtype"] == "c64" else torch.float64
    v = torch.randn(1 << case["n"], 2, generator=gen, device="cuda", dtype=dt)
    v /= math.sqrt(2.0 * (1 << case["n"]))
    return torch.view_as_complex(v)


def _dtype(case):
    return sv.C64 if case["dtype"] == "c64" else sv.C128


def prepare(case, seed):
    s = dict(case)
    ham = _hamiltonian(case, seed)
    if ham is not None:
        s["paulis"], s["coeffs"] = sv.hamiltonian_arrays(ham)
    if case["kind"] == "batch":
        s["circs"], s["params"] = _batch(case, seed)
        return s
    if case["kind"] == "chunk":
        s["state"] = _chunk_state(case, seed)
        return s
    s["circ"] = _circuit(case, seed)
    s["params"] = _params(case, s["circ"].nparams, seed)
    s["sim"] = sv.StateVector(case["n"], case["g"], _dtype(case))
    if case["kind"] in ("grad", "step"):
        s["sim"].ensure_lambda()
    if case["kind"] == "grad":
        dt = torch.float32 if case["dtype"] == "c64" else torch.float64
        s["params"] = torch.tensor(s["params"], dtype=dt, device="cuda", requires_grad=True)
    return s


# ------------------------------------------------------------------ passes --

def _row(case, *values):
    """The pass's numbers in the precision of its state."""
    row = np.concatenate([np.atleast_1d(v) for v in values])
    return row.astype(np.float32 if case["dtype"] == "c64" else np.float64)


def _logical(sim):
    """The state in logical qubit order: a view of its buffer (runs of index
    bits that stand together stay one dimension)."""
    l2p = sim.permutation()
    runs = []                                     # (lowest physical bit, bits), from the highest logical bit down
    for q in range(sim.n - 1, -1, -1):
        if runs and runs[-1][0] == l2p[q] + 1:
            runs[-1] = (int(l2p[q]), runs[-1][1] + 1)
        else:
            runs.append((int(l2p[q]), 1))
    return torch.as_strided(sim.state, [1 << b for _, b in runs], [1 << p for p, _ in runs])


def run(s):
    kind, sched = s["kind"], SCHEDULES[s["schedule"]]
    if kind == "batch":
        e, g, _, _ = sv.batch_run(s["n"], _dtype(s), s["circs"], s["params"], paulis=s["paulis"], coeffs=s["coeffs"])
        return {"energies": _row(s, e), "grads": _row(s, *g)}
    if kind == "chunk":
        e, terms = sv.expect_noalloc(s["state"], s["n"], _dtype(s), s["paulis"], s["coeffs"])
        return {"terms": _row(s, e, terms)}
    sim = s["sim"]
    if kind == "grad":
        e = vqe_energy(s["params"], sim, s["circ"], (s["paulis"], s["coeffs"]), sched, _init(s))
        (g,) = torch.autograd.grad(e, s["params"])
        return {"grad": torch.cat([e.detach().reshape(1), g])}
    if kind == "step":
        e, g, terms = sim.vqe_step(_init(s), s["circ"], s["params"], schedule=sched, paulis=s["paulis"],
                                   coeffs=s["coeffs"], per_term=True)
        return {"terms": _row(s, e, terms), "grad": _row(s, g)}
    sim.reset(_init(s))
    sim.apply_circuit(s["circ"], s["params"], sched)
    if kind == "qsu":
        return {"state": _logical(sim), "layout": sim.permutation()}
    e, terms = sim.expect(schedule=sched, paulis=s["paulis"], coeffs=s["coeffs"])
    return {"terms": _row(s, e, terms)}


# -------------------------------------------------------------------- work --

# real operations per amplitude of one gate (a dense k-qubit matrix: 8 per entry of its row)
_GATE_FLOPS = {W.RY: 6, W.RZ: 6, W.CZ: 0.25, W.GIVENS: 3, W.DEXC: 0.75, W.MAT1: 16, W.MAT2: 32, W.MAT4: 128}


def _gate_flops(circ):
    return sum(_GATE_FLOPS[int(k)] for k in circ.kinds)


def work(case):
    """Bytes: the state vectors a pass cannot do without, psi written once by
    the circuit and read once by the strings; with a gradient also lambda,
    written once, and both read once by the reverse sweep.  Operations: the
    gates (three times with a gradient: psi, then psi and lambda back, and the
    generators' inner products), 3 per amplitude and string for an expectation
    value, 4 for lambda."""
    n, amp = case["n"], 8 if case["dtype"] == "c64" else 16
    size = float(1 << n)
    if case["kind"] == "batch":
        circs, _ = _batch(case, 0)
        gates = sum(_gate_flops(c) for c in circs)
        return {"bytes": 5 * size * amp * case["count"],
                "flops": size * (4 * gates + 4.0 * case["nterms"] * case["count"])}
    if case["kind"] == "chunk":
        return {"bytes": size * amp, "flops": 3.0 * size * case["nterms"]}
    gates = _gate_flops(_circuit(case, 0))
    if case["kind"] == "qsu":
        return {"bytes": size * amp, "flops": size * gates}
    if case["kind"] == "energy":
        return {"bytes": 2 * size * amp, "flops": size * (gates + 3.0 * case["nterms"])}
    per = 4.0 if case["kind"] == "grad" else 7.0
    return {"bytes": 5 * size * amp, "flops": size * (4 * gates + per * case["nterms"])}


# ------------------------------------------------------------------- exact --
# States are [B, 2^n] complex128 tensors: B states that run the same gate list
# with parameters of their own.

def _at(psi, n, bits):
    """View of the amplitudes whose qubits have the given values {q: 0 or 1}."""
    qs = sorted(bits, reverse=True)
    shape, index, above = [psi.shape[0]], [slice(None)], n
    for q in qs:
        shape += [1 << (above - 1 - q), 2]
        index += [slice(None), bits[q]]
        above = q
    return psi.view(shape + [1 << above])[tuple(index)]


def _turn(psi, n, lo, hi, c, s):
    """exp(-i theta Y / 2) on the pair of amplitude sets lo, hi."""
    a, b = _at(psi, n, lo), _at(psi, n, hi)
    form = [psi.shape[0]] + [1] * (a.dim() - 1)
    c, s = c.view(form), s.view(form)
    na = c * a - s * b
    b.copy_(s * a + c * b)
    a.copy_(na)


def _span(kind, qs):
    """The two amplitude sets that a rotation mixes."""
    if kind == W.RY:
        return {qs[0]: 0}, {qs[0]: 1}
    if kind == W.GIVENS:
        return {qs[0]: 1, qs[1]: 0}, {qs[0]: 0, qs[1]: 1}
    return {qs[0]: 1, qs[1]: 1, qs[2]: 0, qs[3]: 0}, {qs[0]: 0, qs[1]: 0, qs[2]: 1, qs[3]: 1}


def _gate(psi, n, circ, i, theta, sign=1.0):
    kind, qs = int(circ.kinds[i]), circ.targets(i)
    if kind == W.CZ:
        _at(psi, n, {qs[0]: 1, qs[1]: 1}).neg_()
    elif kind == W.RZ:
        for bit in (0, 1):
            v = _at(psi, n, {qs[0]: bit})
            v *= torch.exp((0.5j if bit else -0.5j) * sign * theta).view([-1] + [1] * (v.dim() - 1))
    elif kind in (W.RY, W.GIVENS, W.DEXC):
        _turn(psi, n, *_span(kind, qs), torch.cos(0.5 * theta), sign * torch.sin(0.5 * theta))
    else:                                          # a dense matrix: index bit t is target t
        dim = 1 << len(qs)
        at = 2 * int(circ.mat[i])
        u = torch.from_numpy(circ.mats[at:at + 2 * dim * dim].reshape(dim, dim, 2).copy()).to(psi.device)
        parts = [_at(psi, n, {q: j >> t & 1 for t, q in enumerate(qs)}) for j in range(dim)]
        v = torch.view_as_complex(u) @ torch.stack([p.reshape(-1) for p in parts])
        for p, row in zip(parts, v):
            p.copy_(row.view(p.shape))


def _run_circuit(n, circ, params, init, device):
    psi = torch.zeros(params.shape[0], 1 << n, dtype=torch.complex128, device=device)
    psi[:, init] = 1.0
    for i in range(circ.m):
        _gate(psi, n, circ, i, params[:, int(circ.param[i])] if circ.param[i] >= 0 else None)
    return psi


def _signs(n, z, device):
    """(-1)^{|c & z|} over all c as the two factors of its upper and lower half."""
    half = n // 2
    out = []
    for bits, m in ((n - half, z >> half), (half, z & ((1 << half) - 1))):
        v = torch.ones(1, dtype=torch.float64, device=device)
        for b in range(bits):
            v = torch.cat([v, -v if m >> b & 1 else v])
        out.append(v)
    return out


def _moved(v, n, x):
    """v[b ^ x] for every b, v as [B, upper half, lower half]."""
    half = n // 2
    up, low = (torch.arange(k, device=v.device) for k in v.shape[1:])
    if x >> half:
        v = v.index_select(1, up ^ (x >> half))
    return v.index_select(2, low ^ (x & ((1 << half) - 1))) if x & ((1 << half) - 1) else v


def _split(v, n):
    return v.view(v.shape[0], 1 << (n - n // 2), 1 << (n // 2))


def _grouped(paulis):
    """String numbers by their X/Y mask."""
    groups = {}
    for t, (x, z) in enumerate(paulis):
        groups.setdefault(x, []).append((t, z))
    return groups


def _terms(psi, n, paulis):
    """<psi|P_t|psi> for every string t, [nterms] (B = 1): with w[c] =
    conj(psi[c ^ x]) psi[c], i^nY sum_c (-1)^{|c & z|} w[c]."""
    v = _split(psi, n)
    out = torch.zeros(len(paulis), dtype=torch.float64, device=psi.device)
    for x, members in _grouped(paulis).items():
        w = (_moved(v, n, x).conj() * v)[0]
        for k in range(0, len(members), 32):
            part = members[k:k + 32]
            signs = [_signs(n, z, psi.device) for _, z in part]
            low = torch.stack([s[1] for s in signs], 1)
            for odd in (0, 1):
                pick = [j for j, (_, z) in enumerate(part) if bin(x & z).count("1") % 2 == odd]
                if not pick:
                    continue
                sums = ((w.imag if odd else w.real) @ low[:, pick])
                for j, col in zip(pick, sums.t()):
                    t, z = part[j]
                    ny = bin(x & z).count("1") % 4      # i^nY (re + i im), real part
                    sign = (1.0, -1.0, -1.0, 1.0)[ny]
                    out[t] = sign * torch.dot(signs[j][0], col)
    return out


def _h_psi(psi, n, paulis, coeffs):
    """sum_t a_t P_t psi: (P psi)[b] = i^nY (-1)^{|c & z|} psi[c], c = b ^ x."""
    v = _split(psi, n)
    lam = torch.zeros_like(v)
    for x, members in _grouped(paulis).items():
        part = torch.zeros_like(v)
        for t, z in members:
            up, low = _signs(n, z, psi.device)
            ny = bin(x & z).count("1") % 4
            if len(members) == 1:
                part = v * (up * coeffs[t] * 1j ** ny)[:, None] * low[None, :]
            else:
                part.addcmul_(v, ((up * coeffs[t] * 1j ** ny)[:, None] * low[None, :])[None])
        lam += _moved(part, n, x)
    return lam.view(psi.shape)


def _dot(a, b):
    """<a|b> over the amplitudes, [B]."""
    if a.shape[0] == 1:
        return torch.vdot(a.reshape(-1), b.reshape(-1)).reshape(1)
    return (a.conj() * b).reshape(a.shape[0], -1).sum(1)


def _reverse(psi, lam, n, circ, params):
    """dE/dparams, [B, np]: Im <lambda|G_k|psi> per gate, from the last back."""
    grad = torch.zeros(params.shape, dtype=torch.float64, device=psi.device)
    for i in range(circ.m - 1, -1, -1):
        kind, qs, p = int(circ.kinds[i]), circ.targets(i), int(circ.param[i])
        if p >= 0:
            if kind == W.RZ:                       # Z
                v = [_dot(_at(lam, n, {qs[0]: b}), _at(psi, n, {qs[0]: b})) for b in (0, 1)]
                grad[:, p] += (v[0] - v[1]).imag
            else:                                  # Y on the pair: Im(-i <l0|p1> + i <l1|p0>)
                lo, hi = _span(kind, qs)
                grad[:, p] += (_dot(_at(lam, n, hi), _at(psi, n, lo)) - _dot(_at(lam, n, lo), _at(psi, n, hi))).real
        theta = params[:, p] if p >= 0 else None
        _gate(psi, n, circ, i, theta, -1.0)
        _gate(lam, n, circ, i, theta, -1.0)
    return grad


def _gradient(n, circ, params, init, paulis, coeffs, device):
    """(energies [B], gradients [B, np], the forward state)."""
    psi = _run_circuit(n, circ, params, init, device)
    lam = _h_psi(psi, n, paulis, coeffs)
    e = _dot(psi, lam).real
    return e, psi, lam


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    # the whole-gradient simulation of 1024 strings takes seconds at n = 27, a minute or more at n = 30
    if n > (28 if kind in ("qsu", "energy", "chunk") else 27):
        return None
    device = "cuda" if torch.cuda.is_available() else "cpu"
    ham = _hamiltonian(case, seed)
    if ham is not None:
        xs, zs = W.pauli_masks(ham)
        paulis = [(int(x), int(z)) for x, z in zip(xs, zs)]
        coeffs = [float(c) for c in ham.coeffs]
        weights = torch.tensor(coeffs, dtype=torch.float64, device=device)
    if kind == "batch":
        circs, plist = _batch(case, seed)
        energies = torch.zeros(len(circs), dtype=torch.float64, device=device)
        grads = [None] * len(circs)
        for m in sorted({c.m for c in circs}):
            same = [b for b, c in enumerate(circs) if c.m == m]
            params = torch.from_numpy(np.stack([plist[b] for b in same])).to(device)
            e, psi, lam = _gradient(n, circs[same[0]], params, 0, paulis, coeffs, device)
            g = _reverse(psi, lam, n, circs[same[0]], params)
            energies[same] = e
            for b, row in zip(same, g):
                grads[b] = row
        return {"energies": energies, "grads": torch.cat(grads)}
    if kind == "chunk":
        psi = _chunk_state(case, seed).to(torch.complex128).view(1, -1)
        terms = _terms(psi, n, paulis)
        return {"terms": torch.cat([torch.dot(weights, terms).reshape(1), terms])}
    circ = _circuit(case, seed)
    params = torch.from_numpy(_params(case, circ.nparams, seed)).to(device).view(1, -1)
    if kind in ("qsu", "energy"):
        psi = _run_circuit(n, circ, params, _init(case), device)
        if kind == "qsu":
            return {"state": psi.view(-1), "layout": None}
        terms = _terms(psi, n, paulis)
        return {"terms": torch.cat([torch.dot(weights, terms).reshape(1), terms])}
    e, psi, lam = _gradient(n, circ, params, _init(case), paulis, coeffs, device)
    if kind == "grad":
        return {"grad": torch.cat([e, _reverse(psi, lam, n, circ, params)[0]])}
    terms = _terms(psi, n, paulis)
    return {"terms": torch.cat([torch.dot(weights, terms).reshape(1), terms]),
            "grad": _reverse(psi, lam, n, circ, params)[0]}
