"""Passes full of RYs whose factors (the larger of cos and sin of the half
angle, taken out of the rotation) are as small as they come: with angles at odd
multiples of pi/2 each is 2^-1/2, 2^-128 over 256 of them.

Bounds: a rotation adds at most about 4 u to the state's error norm, 256 of
them in random directions 64 u = 4e-6, so 2e-5 for amplitudes and 2e-5 l1 for
energies and gradients as in the other complex64 tests."""
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

KINDS = {"rotations": (W.RY,), "diagonal": (W.RY, W.RY, W.RY, W.RZ, W.CZ), "mixed": (W.RY, W.RY, W.RY, W.GIVENS),
         "matrix": (W.RY, W.RY, W.RY, W.MAT1)}


def circuit(n, m, kinds, seed):
    c = W.random_circuit(n, m, seed, kinds)
    one = np.flatnonzero(np.asarray(c.kinds) == W.MAT1)
    c.mats = W.random_unitary_mats(len(one), 2, seed) if len(one) else np.zeros(0)
    for j, i in enumerate(one):
        c.mat[i] = 4 * j
    return c


def angles(c, seed):
    """Odd multiples of pi/2: every RY keeps a factor of 2^-1/2, of either sign."""
    rng = np.random.default_rng(seed)
    return math.pi / 2 * rng.choice([-3.0, -1.0, 1.0, 3.0, 5.0], c.nparams)


# one tile of the smallest and of the largest size, several tiles
@pytest.mark.parametrize("n,tile", [(9, 9), (13, 0), (14, 0)])
@pytest.mark.parametrize("m", [48, 130, 256])
@pytest.mark.parametrize("kinds", sorted(KINDS))
def test_small_factors(kinds, m, n, tile):
    c = circuit(n, m, KINDS[kinds], 7 * m + n)
    params = angles(c, n + m)
    h = W.jw_hamiltonian(n, 24, 9)
    l1 = float(np.abs(h.coeffs).sum())
    o = sv.default_options(sv.C64)
    if tile:
        o.tile_bits, o.low_bits = tile, 3
    s = sv.StateVector(n, 0, sv.C64, options=o)
    s.reset(6)
    s.apply_circuit(c, params, sv.LAZY)
    ref = oracle.apply_circuit(oracle.basis_state(n, 6), c, params)
    assert np.max(np.abs(s.get_state() - ref)) < 2e-5
    s.reset(6)
    e, g = s.grad(c, params, h, sv.LAZY)
    assert abs(e - ograd.objective(c, params, h, 6)) < 2e-5 * l1
    which = list(range(0, c.nparams, max(1, c.nparams // 8)))
    fd = ograd.finite_difference(c, params, h, 6, which=which)
    assert np.max(np.abs(g[which] - fd[which])) < 2e-5 * l1


@pytest.mark.parametrize("n", [13, 14])
def test_small_factors_in_a_batch(n):
    circs = [circuit(n, m, KINDS[k], m) for k, m in (("rotations", 256), ("diagonal", 130), ("mixed", 200))]
    params = [angles(c, i) for i, c in enumerate(circs)]
    h = W.jw_hamiltonian(n, 24, 9)
    l1 = float(np.abs(h.coeffs).sum())
    e, g, _, _ = sv.batch_run(n, sv.C64, circs, params, h, init_index=3)
    wide = sv.StateVector(n, 0, sv.C128)
    for b, c in enumerate(circs):
        wide.reset(3)
        e1, g1 = wide.grad(c, params[b], h, sv.LAZY)
        assert abs(e1 - ograd.objective(c, params[b], h, 3)) < 1e-10
        assert abs(e[b] - e1) < 2e-5 * l1
        assert np.max(np.abs(np.asarray(g[b]) - g1)) < 2e-5 * l1
