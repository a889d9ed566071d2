"""H|psi>, expectation values and gradients of states so small that one run
holds them (a coset span of dimension 0: complex128 below 8 qubits, and any
state when the options ask for long runs), against the FP64 oracle.  Bounds as
for the other coset tests: 1e-5 and 1e-12 per string; an element of H|psi> at
most 2 T u l1 with T = 32; gradients 2e-5 l1 and 1e-7 (finite differences)."""
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


@pytest.mark.parametrize("dtype", [sv.C64, sv.C128])
@pytest.mark.parametrize("n,g,run", [(4, 0, 0), (5, 1, 0), (6, 0, 0), (6, 2, 0), (7, 0, 0), (7, 3, 0), (8, 1, 0), (9, 0, 0),
                                     (10, 0, 10), (9, 0, 9)])
@pytest.mark.parametrize("ham", ["random", "jw"])
def test_states_of_one_run(dtype, n, g, run, ham):
    h = W.random_hamiltonian(n, 24, 3) if ham == "random" else W.jw_hamiltonian(n, 24, 3)
    l1 = float(np.abs(h.coeffs).sum())
    o = sv.default_options(dtype)
    if run:
        o.evc_low_bits, o.evc_span = run, 0
    rng = np.random.default_rng(n)
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dtype == sv.C64 else np.complex128)
    wide = psi.astype(np.complex128)
    ref = oracle.expect_terms(wide, h).real
    s = sv.StateVector(n, g, dtype, options=o)
    s.set_state(psi)
    _, pt = s.expect(h, sv.LAZY)
    assert np.max(np.abs(pt - ref)) < (1e-5 if dtype == sv.C64 else 1e-12)
    s.set_state(psi)
    e, lam = s.apply_hamiltonian(h)
    vtol = 64 * l1 * (2.0 ** -24 if dtype == sv.C64 else 2.0 ** -53)
    assert np.max(np.abs(lam.cpu().numpy().astype(np.complex128) - oracle.apply_hamiltonian(wide, h))) < vtol
    assert abs(e - float(np.dot(h.coeffs, ref))) < (1e-5 if dtype == sv.C64 else 1e-12) * l1
    c = W.hea_circuit(n, 2)
    params = W.uniform_params(c.nparams, 4, -2, 2)
    s.reset(3)
    _, got = s.grad(c, params, h, sv.LAZY)
    which = list(range(0, c.nparams, max(1, c.nparams // 6)))
    fd = ograd.finite_difference(c, params, h, 3, which=which)
    assert np.max(np.abs(got[which] - fd[which])) < (1e-7 if dtype == sv.C128 else 2e-5 * l1)


@pytest.mark.parametrize("dtype,n", [(sv.C64, 20), (sv.C64, 21), (sv.C128, 18), (sv.C128, 19)])
def test_hamiltonian_passes_of_both_kinds(dtype, n):
    # one mask with many strings and eleven with one: passes in slices and of whole cosets in one call
    rng = np.random.default_rng(n)
    x = [rng.random(n) < 0.4 for _ in range(12)]
    rows = [np.where(x[0], rng.choice([W.PX, W.PY], n), rng.choice([0, W.PZ], n)) for _ in range(60)]
    rows += [np.where(m, rng.choice([W.PX, W.PY], n), rng.choice([0, W.PZ], n)) for m in x[1:]]
    h = W.Hamiltonian(n, np.array(rows, np.uint8), np.linspace(-1.0, 1.0, len(rows)))
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dtype == sv.C64 else np.complex128)
    wide = psi.astype(np.complex128)
    l1 = float(np.abs(h.coeffs).sum())
    for order in (slice(None), slice(None, None, -1)):
        part = W.Hamiltonian(n, h.letters[order], h.coeffs[order])
        s = sv.StateVector(n, 0, dtype)
        s.set_state(psi)
        e, lam = s.apply_hamiltonian(part)
        vtol = 2 * len(rows) * l1 * (2.0 ** -24 if dtype == sv.C64 else 2.0 ** -53) * float(np.max(np.abs(psi)))
        assert np.max(np.abs(lam.cpu().numpy().astype(np.complex128) - oracle.apply_hamiltonian(wide, part))) < vtol
        ref = float(np.dot(part.coeffs, oracle.expect_terms(wide, part).real))
        assert abs(e - ref) < (1e-5 if dtype == sv.C64 else 1e-12) * l1
