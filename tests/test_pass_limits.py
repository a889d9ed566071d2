"""Gate passes with more register phases than their tables have room for.

A phase takes about a kilobyte of tables beside 128 KB of tiles, so a pass of
up to 256 gates on few qubits can need more than a block's shared memory; it
is then cut into passes over the same staged bits.

Bounds, u = 2^-24 or 2^-53.  A dense or pair gate adds at most about 8 u to the
state's error norm, 256 of them in random directions sqrt(256) 8 u = 8e-6
(2e-14), so amplitudes to 2e-5 and 1e-12 as in the other gate tests; gradients
against central differences as there, 2e-5 l1 and 1e-7."""
import math

import numpy as np
import pytest

import oracle
from oracle import grad as ograd
from paper_2410_04252_gb300 import workloads as W

sv = pytest.importorskip("paper_2410_04252_gb300.sv")
torch = pytest.importorskip("torch")

MATRICES = (W.MAT1, W.MAT2, W.MAT4)


def circuit(n, m, kinds, seed):
    c = W.random_circuit(n, m, seed, kinds)
    offset, mats = 0, []
    for i in range(c.m):
        if int(c.kinds[i]) in MATRICES:
            dim = 1 << W.GATE_NQ[int(c.kinds[i])]
            mats.append(W.random_unitary_mats(1, dim, seed * 1000 + i))
            c.mat[i] = offset
            offset += dim * dim
    c.mats = np.concatenate(mats) if mats else np.zeros(0)
    return c


# gate kinds, count, and whether a complex64 pass of 2^13 amplitudes must be cut
CASES = [
    ((W.MAT4,), 80, False), ((W.MAT4,), 120, True), ((W.MAT4,), 256, True),
    ((W.MAT2,), 180, False), ((W.MAT2,), 256, True),
    ((W.GIVENS,), 150, False), ((W.GIVENS,), 256, True),
    ((W.DEXC,), 60, False), ((W.DEXC,), 256, True),
    ((W.RY, W.RZ, W.CZ, W.GIVENS, W.DEXC), 256, True),
    ((W.RY, W.RZ, W.CZ), 256, False),
]


@pytest.mark.parametrize("kinds,m,cut", CASES)
def test_long_passes_are_cut(kinds, m, cut):
    c = circuit(13, m, kinds, 70 + m)
    plan = sv.plan_qsu(13, 0, c, sv.LAZY)
    assert (len(plan["passes"]) > 1) == cut
    assert len({p["bits"] for p in plan["passes"]}) == 1
    order = [u for p in plan["passes"] for u in p["ops"]]
    assert sorted(order) == list(range(m))
    if not {W.RZ, W.CZ} & set(kinds):      # (diagonal gates commute among each other)
        last = [-1] * 13                   # gates that share a qubit keep their order
        for u in order:
            assert all(last[q] < u for q in c.targets(u))
            for q in c.targets(u):
                last[q] = u


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("dtype,n", [(sv.C64, 13), (sv.C128, 12), (sv.C64, 15)])
@pytest.mark.parametrize("kinds,m", [c[:2] for c in CASES])
def test_long_passes_run(kinds, m, dtype, n):
    c = circuit(n, m, kinds, 70 + m)
    params = W.uniform_params(c.nparams, 5 + m, -2, 2)
    ref = oracle.apply_circuit(oracle.basis_state(n, 5), c, params)
    s = sv.StateVector(n, 0, dtype)
    s.reset(5)
    s.apply_circuit(c, params, sv.LAZY)
    assert np.max(np.abs(s.get_state() - ref)) < (2e-5 if dtype == sv.C64 else 1e-12)
    h = W.jw_hamiltonian(n, 24, 9)
    l1 = float(np.abs(h.coeffs).sum())
    s.reset(6)
    e, got = s.grad(c, params, h, sv.LAZY)
    assert abs(e - ograd.objective(c, params, h, 6)) < (1e-10 if dtype == sv.C128 else 2e-5 * l1)
    if c.nparams:
        which = list(range(0, c.nparams, max(1, c.nparams // 4)))
        fd = ograd.finite_difference(c, params, h, 6, which=which)
        assert np.max(np.abs(got[which] - fd[which])) < (1e-7 if dtype == sv.C128 else 2e-5 * l1)
