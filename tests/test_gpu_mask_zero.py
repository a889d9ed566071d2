"""Strings without X and Y (the mask 0: |psi|^2 with signs), alone and among
others, in the numbers at which complex128 groups of four, the groups a mask is split into
(256 strings) and the choice between slices and whole cosets change.  Bounds as for the other expectation tests:
1e-5 and 1e-12."""
import numpy as np
import pytest

import oracle
from paper_2410_04252_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
sv = pytest.importorskip("paper_2410_04252_gb300.sv")


# fewer staged bits than the state's, one coset, both sides of the lines of both types
@pytest.mark.parametrize("dtype,n", [(sv.C64, 8), (sv.C64, 13), (sv.C64, 17), (sv.C64, 20), (sv.C64, 22),
                                     (sv.C128, 8), (sv.C128, 12), (sv.C128, 18), (sv.C128, 19), (sv.C128, 20)])
@pytest.mark.parametrize("zeros,others", [(1, 0), (3, 0), (4, 30), (5, 9), (47, 0), (200, 60), (300, 0), (300, 40)])
def test_mask_zero(dtype, n, zeros, others):
    rng = np.random.default_rng(100 * n + zeros)
    z = np.unique((rng.random((zeros, n)) < 0.4) * W.PZ, axis=0).astype(np.uint8)
    letters = np.concatenate([z, W.jw_hamiltonian(n, others, 5).letters]) if others else z
    letters = letters[rng.permutation(len(letters))]
    h = W.Hamiltonian(n, letters, np.linspace(-1.0, 1.0, len(letters)))
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dtype == sv.C64 else np.complex128)
    ref = oracle.expect_terms(psi.astype(np.complex128), h).real
    tol = 1e-5 if dtype == sv.C64 else 1e-12
    s = sv.StateVector(n, min(2, n - 4), dtype)
    for sched in (sv.LAZY, sv.DIRECT) + ((sv.EAGER,) if zeros < 50 else ()):
        s.set_state(psi)
        _, pt = s.expect(h, sched)
        assert np.max(np.abs(pt - ref)) < tol
    if len(letters) <= 256:
        s.set_state(psi)
        p, c = sv.hamiltonian_arrays(h)
        _, pt = sv.expect_noalloc(s.state, n, dtype, p, c)
        assert np.max(np.abs(pt - ref)) < tol
