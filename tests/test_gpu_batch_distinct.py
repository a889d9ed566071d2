"""A batch whose states all have circuits of their own (planned on several host
threads), among them passes that are cut because their tables exceed the room
beside the batched kernel's tiles, against the single-state complex128 path.
Bounds as in the other batch tests: 2e-5 l1."""
import numpy as np
import pytest

from oracle import grad as ograd
from paper_2410_04252_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
sv = pytest.importorskip("paper_2410_04252_gb300.sv")


@pytest.mark.parametrize("n,dtype", [(12, sv.C64), (13, sv.C64), (14, sv.C64), (12, sv.C128)])
@pytest.mark.parametrize("count", [3, 40])
def test_distinct_circuits(n, dtype, count):
    kinds = [(W.GIVENS,), (W.RY, W.CZ), (W.DEXC, W.GIVENS), (W.RY, W.RZ, W.CZ, W.GIVENS, W.DEXC)]
    circs = [W.random_circuit(n, 40 + 220 * (i % 5 == 0), 11 * i + 1, kinds[i % 4]) for i in range(count)]
    params = [W.uniform_params(c.nparams, i, -2, 2) for i, c in enumerate(circs)]
    h = W.jw_hamiltonian(n, 24, 9)
    l1 = float(np.abs(h.coeffs).sum())
    e, g, _, _ = sv.batch_run(n, dtype, circs, params, h, init_index=5)
    wide = sv.StateVector(n, 0, sv.C128)
    tol = 2e-5 * l1 if dtype == sv.C64 else 1e-10 * l1
    for b in range(0, count, max(1, count // 10)):
        wide.reset(5)
        e1, g1 = wide.grad(circs[b], params[b], h, sv.LAZY)
        if b < 3:
            assert abs(e1 - ograd.objective(circs[b], params[b], h, 5)) < 1e-10
        assert abs(e[b] - e1) < tol
        assert np.max(np.abs(np.asarray(g[b]) - g1)) < tol


def test_the_failing_state_is_named():
    circs = [W.random_circuit(13, 20, i, (W.RY, W.CZ)) for i in range(20)]
    params = [np.zeros(c.nparams) for c in circs]
    circs[17] = W.random_circuit(13, 20, 17, (W.RY, W.CZ))
    circs[17].qubits[3, 0] = 13
    with pytest.raises(sv.SvError, match="state 17"):
        sv.batch_run(13, sv.C64, circs, params, W.jw_hamiltonian(13, 8, 1))
