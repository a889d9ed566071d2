"""The variants that a dispatch chooses among by size, type and operations,
each at the edges of its range, against the FP64 oracle.

Bounds, with u = 2^-24 (complex64) or 2^-53 (complex128).  Amplitudes: 2e-5 and
1e-12, as for the other gate tests.  A string's expectation: each thread adds
at most a few tens of products of a coset before FP64 takes over and
sum |psi_i psi_j| <= 1, so 1e-5 (about 160 u) and 1e-12.  An element of
H|psi>: at most T products of T strings, 2 T u l1 max|psi| with T = 128.
Gradients against central differences (step 1e-5): 1e-7 for complex128 as
elsewhere; for complex64 2 |H| |dpsi| with |dpsi| <= 1e-5, 2e-5 l1."""
import math

import numpy as np
import pytest

import oracle
from oracle import grad as ograd
from paper_2410_04252_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
sv = pytest.importorskip("paper_2410_04252_gb300.sv")

AMP_TOL = {sv.C64: 2e-5, sv.C128: 1e-12}
TERM_TOL = {sv.C64: 1e-5, sv.C128: 1e-12}
UNIT = {sv.C64: 2.0 ** -24, sv.C128: 2.0 ** -53}
KINDS = {
    "diagonal": (W.RY, W.RZ, W.CZ),
    "pairs": (W.GIVENS, W.DEXC),
    "mixed": (W.RY, W.RZ, W.CZ, W.GIVENS, W.DEXC),
    "matrices": (W.RY, W.CZ, W.GIVENS, W.MAT1, W.MAT2, W.MAT4),
}


def circuit(n, m, seed, kinds):
    c = W.random_circuit(n, m, seed, KINDS[kinds])
    offs, mats = 0, []
    for i in range(c.m):
        k = int(c.kinds[i])
        if k in (W.MAT1, W.MAT2, W.MAT4):
            dim = 1 << W.GATE_NQ[k]
            mats.append(W.random_unitary_mats(1, dim, seed * 1000 + i))
            c.mat[i] = offs
            offs += dim * dim
    c.mats = np.concatenate(mats) if mats else np.zeros(0)
    return c


def random_state(n, seed):
    rng = np.random.default_rng(seed)
    v = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    return v / np.linalg.norm(v)


@pytest.mark.parametrize("dtype", [sv.C64, sv.C128])
@pytest.mark.parametrize("kinds", sorted(KINDS))
# below the register phases, their smallest and largest tile, one tile, many tiles and a swap
@pytest.mark.parametrize("n,g,tile", [(8, 0, 8), (9, 0, 9), (12, 2, 10), (13, 0, 0), (17, 3, 0)])
def test_gate_step_kinds(dtype, kinds, n, g, tile):
    c = circuit(n, 90, 31 + n, kinds)
    params = W.uniform_params(c.nparams, 5 + n, -math.pi, math.pi)
    o = sv.default_options(dtype)
    if tile:
        o.tile_bits, o.low_bits = tile, 3
    ref = oracle.apply_circuit(oracle.basis_state(n, 5), c, params)
    for sched in (sv.LAZY, sv.EAGER):
        s = sv.StateVector(n, g, dtype, options=o)
        s.reset(5)
        s.apply_circuit(c, params, sched)
        assert np.max(np.abs(s.get_state() - ref)) < AMP_TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.C64, sv.C128])
@pytest.mark.parametrize("kinds", sorted(KINDS))
@pytest.mark.parametrize("n,g,tile", [(9, 0, 9), (14, 3, 0)])
def test_adjoint_step_kinds(dtype, kinds, n, g, tile):
    c = circuit(n, 60, 53 + n, kinds)
    params = W.uniform_params(c.nparams, 7 + n, -2, 2)
    h = W.jw_hamiltonian(n, 24, 9)
    l1 = float(np.abs(h.coeffs).sum())
    which = list(range(0, c.nparams, max(1, c.nparams // 6)))
    fd = ograd.finite_difference(c, params, h, 6, which=which)
    o = sv.default_options(dtype)
    if tile:
        o.tile_bits, o.low_bits = tile, 3
    s = sv.StateVector(n, g, dtype, options=o)
    s.reset(6)
    e, got = s.grad(c, params, h, sv.LAZY)
    assert abs(e - ograd.objective(c, params, h, 6)) < (1e-10 if dtype == sv.C128 else 2e-5 * l1)
    assert np.max(np.abs(got[which] - fd[which])) < (1e-7 if dtype == sv.C128 else 2e-5 * l1)


def hamiltonian(kind, n):
    if kind == "jw":            # about four strings a mask
        return W.jw_hamiltonian(n, 96, 400 + n)
    if kind == "pairs":         # every X/Y form of a few masks, bit 0 and neighbours among them
        letters = []
        for i, j in ((0, 1), (0, n - 1), (1, 2), (2, n - 2), (n - 2, n - 1)):
            for p in (W.PX, W.PY):
                for q in (W.PX, W.PY):
                    row = np.zeros(n, np.uint8)
                    row[i], row[j] = p, q
                    row[i + 1:j] = W.PZ
                    letters.append(row)
        return W.Hamiltonian(n, np.array(letters), np.linspace(-1.0, 1.0, len(letters)))
    h = W.random_hamiltonian(n, 12, 300 + n)
    # an identity, a pure Z, X and Y on qubit 0 alone, and two products of other strings' masks
    extra = np.zeros((6, n), np.uint8)
    extra[1, n - 1] = W.PZ
    extra[2, 0] = W.PX
    extra[3, 0] = W.PY
    flip = np.isin(h.letters, (W.PX, W.PY))
    extra[4] = np.where(flip[0] ^ flip[1], W.PY, 0)
    extra[5] = np.where(flip[2] ^ flip[3], W.PX, W.PZ)
    return W.Hamiltonian(n, np.concatenate([h.letters, extra]), np.concatenate([h.coeffs, np.linspace(-1, 1, 6)]))


@pytest.mark.parametrize("kind", ["jw", "pairs", "random"])
# fewer cosets than CTAs, both sides of the line to whole cosets, several cosets a CTA
@pytest.mark.parametrize("dtype,n", [(sv.C64, 5), (sv.C64, 13), (sv.C64, 20), (sv.C64, 21), (sv.C64, 22),
                                     (sv.C128, 5), (sv.C128, 14), (sv.C128, 18), (sv.C128, 19), (sv.C128, 21)])
def test_coset_pass_variants(dtype, n, kind):
    h = hamiltonian(kind, n)
    l1 = float(np.abs(h.coeffs).sum())
    psi = random_state(n, n).astype(np.complex64 if dtype == sv.C64 else np.complex128)
    wide = psi.astype(np.complex128)
    ref = oracle.expect_terms(wide, h).real
    refv = oracle.apply_hamiltonian(wide, h)
    vtol = 256 * UNIT[dtype] * l1 * float(np.max(np.abs(psi)))
    for g in (0, min(2, n - 4)):
        s = sv.StateVector(n, g, dtype)
        s.set_state(psi)
        e, pt = s.expect(h, sv.LAZY)
        assert np.max(np.abs(pt - ref)) < TERM_TOL[dtype]
        assert abs(e - float(np.dot(h.coeffs, ref))) < TERM_TOL[dtype] * l1
    s = sv.StateVector(n, 0, dtype)
    s.set_state(psi)
    e, lam = s.apply_hamiltonian(h)
    assert list(s.permutation()) == list(range(n))
    assert np.max(np.abs(lam.cpu().numpy().astype(np.complex128) - refv)) < vtol
    assert abs(e - float(np.dot(h.coeffs, ref))) < TERM_TOL[dtype] * l1
    paulis, coeffs = sv.hamiltonian_arrays(h)
    e, pt = sv.expect_noalloc(s.state, n, dtype, paulis, coeffs)
    assert np.max(np.abs(pt - ref)) < TERM_TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.C64, sv.C128])
@pytest.mark.parametrize("n", [1, 2, 11, 20])
def test_reset_to_a_basis_state(dtype, n):
    for g in {0, min(2, max(0, n - 4))}:
        s = sv.StateVector(n, g, dtype)
        for index in {0, 1, (1 << n) - 1, (1 << n) // 2}:
            s.reset(index)
            got = s.get_state()
            assert got[index] == 1 and np.count_nonzero(got) == 1


@pytest.mark.parametrize("n", [12, 13, 14])
def test_batch_step_loops(n):
    # gate by gate (12), one tile (13), several tiles and passes (14); kinds mixed in one batch
    circs, params = [], []
    for i, kinds in enumerate(("diagonal", "pairs", "mixed", "diagonal")):
        c = circuit(n, 70 - 30 * (i == 3), 90 + i, kinds)
        circs.append(c)
        params.append(W.uniform_params(c.nparams, 3 + i, -2, 2))
    circs.append(W.hea_circuit(n, 3))
    params.append(W.uniform_params(circs[-1].nparams, 9, 0.0, 2 * math.pi))
    ham = W.jw_hamiltonian(n, 40, 12)
    l1 = float(np.abs(ham.coeffs).sum())
    e, g, t, st = sv.batch_run(n, sv.C64, circs, params, ham, init_index=3)
    wide = sv.StateVector(n, 0, sv.C128)
    for b, c in enumerate(circs):
        wide.reset(3)
        e1, g1 = wide.grad(c, params[b], ham, sv.LAZY)
        assert abs(e1 - ograd.objective(c, params[b], ham, 3)) < 1e-10
        assert abs(e[b] - e1) < 2e-5 * l1
        assert np.max(np.abs(np.asarray(g[b]) - g1)) < 2e-5 * l1
