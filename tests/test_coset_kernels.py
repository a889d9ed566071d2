"""The expectation kernels for few strings and for masks of one or two staged
bits, on strings that are known to reach them: every place of a string in the
plan (which register bit flips, whether bit 0 flips too, real or imaginary
part, partners read) occurs in a set here, and the sets' passes are checked to
run in the kernel meant.

Bounds as for the other expectation tests: each thread adds at most a few tens
of products of a coset before FP64 takes over and sum |psi_i psi_j| <= 1, so
1e-5 (about 160 u) and 1e-12."""
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2410_04252_gb300 import workloads as W

sv = pytest.importorskip("paper_2410_04252_gb300.sv")
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_2410_04252_gb300")


@pytest.fixture(scope="module")
def plan_of(tmp_path_factory):
    """passes(h, g, dtype): per pass the codes of its unit items and of its
    register phases' items, and the groups left to the general kernels."""
    exe = str(tmp_path_factory.mktemp("plan") / "coset_plan")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(PKG, "csrc"), "-o", exe,
                           os.path.join(HERE, "coset_plan.cpp"), os.path.join(PKG, "_build", "libsv.so"),
                           "-Wl,-rpath," + os.path.join(PKG, "_build")])

    def passes(h, g, dtype):
        p, _ = sv.hamiltonian_arrays(h)
        text = f"{h.n} {g} {int(dtype == sv.C128)} {len(p)}\n" + "\n".join(f"{int(x)} {int(z)}" for x, z in p)
        out = []
        for line in subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines():
            w = line.split()
            u, r, e = w.index("unit"), w.index("phases"), w.index("rest")
            out.append(dict(strings=int(w[3]), unit=[int(v) for v in w[u + 1:r]],
                            phases=[int(v) for v in w[r + 1:e]], rest=int(w[e + 1])))
        return out

    return passes


def hamiltonian(n, strings):
    letters = np.zeros((len(strings), n), np.uint8)
    for i, (x, z) in enumerate(strings):
        for q in range(n):
            letters[i, q] = (0, W.PZ, W.PX, W.PY)[2 * (x >> q & 1) + (z >> q & 1)]
    return W.Hamiltonian(n, letters, np.linspace(-1.0, 1.0, len(strings)))


def odd_y(rng, n, x, odd):
    """A random z with an odd or even number of Y letters on x."""
    z = int(rng.integers(0, 1 << n))
    if bin(x & z).count("1") % 2 != odd:
        z ^= x & -x
    return z


def few(n, seed, products):
    """Eight independent masks, on both sides of every choice bit 0 and the
    part, and `products` masks inside their span."""
    rng = np.random.default_rng(seed)
    masks = [(int(rng.integers(1, 1 << n)) & ~1) | 1 << (n - 1 - i) | (i + seed) % 2 for i in range(8)]
    masks = [m & ~sum(1 << (n - 1 - j) for j in range(8) if j != i) for i, m in enumerate(masks)]
    masks += [masks[i % 8] ^ masks[(i + 3) % 8] ^ (masks[(i + 5) % 8] if i % 3 == 0 else 0) for i in range(products)]
    return hamiltonian(n, [(m, odd_y(rng, n, m, (i // 2 + seed // 2) % 2)) for i, m in enumerate(masks)])


def neighbours(n, seed, bits, singles, forms):
    """Masks of two of the given qubits (a ring and its chords) and of one, the
    first `forms` of the four X/Y forms each, random Z elsewhere."""
    rng = np.random.default_rng(seed)
    k = len(bits)
    masks = [1 << bits[i] | 1 << bits[(i + d) % k] for d in (1, 2) for i in range(k)]
    masks += [1 << b for b in bits[:singles]]
    return hamiltonian(n, [(m, odd_y(rng, n, m, f % 2) ^ (m if f >= 2 else 0)) for m in dict.fromkeys(masks)
                           for f in range(forms)])


FEW = [(0, 0), (1, 0), (2, 3), (3, 5), (4, 8), (5, 1)]          # seed, products
PAIRS = [(0, (0, 1, 2, 3, 4, 5), 6, 4), (1, (0, 4, 5, 9, 21, 20), 0, 4), (2, (1, 7, 12, 15, 18), 5, 3),
         (3, (2, 3, 10, 13, 16, 19, 20), 2, 2), (4, (3, 6, 8, 9, 11, 14, 17, 20), 8, 1)]


def few_cases(n):
    return [few(n, *c) for c in FEW]


def pair_cases(n):
    return [neighbours(n, s, [b - (22 - n) if b > 18 else b for b in bits], k, f) for s, bits, k, f in PAIRS]


def test_every_place_is_reached(plan_of):
    codes = set()
    for h in few_cases(22):
        for p in plan_of(h, 0, sv.C64):
            codes |= set(p["unit"])
            assert p["unit"] and not p["phases"] and not p["rest"]
    assert codes == set(range(18))
    for dtype, n in ((sv.C64, 22), (sv.C128, 21)):
        kinds = set()
        for h in pair_cases(n):
            ps = plan_of(h, 0, dtype)
            assert any(p["phases"] for p in ps)
            kinds |= {c for p in ps for c in p["phases"]}
        # places of (h, l), then of single bits: 10 + h
        two = {c for c in kinds if c < 10}
        one = {c for c in kinds if c >= 10}
        assert len(two) == (10 if dtype == sv.C64 else 6) and len(one) == (5 if dtype == sv.C64 else 4)


def test_partner_reading_strings_take_register_phases(plan_of):
    # nine masks of two among nine qubits: no string's mask is a basis vector of its own
    masks = [(1 << (8 + i)) | (1 << (8 + (i + 2) % 9)) for i in range(9)]
    rng = np.random.default_rng(1)
    h = hamiltonian(22, [(m, int(rng.integers(0, 1 << 22))) for m in masks])
    for p in plan_of(h, 0, sv.C64):
        partners = sum(c >= 16 for c in p["unit"])
        assert not (p["unit"] and p["phases"])
        assert 2 * partners <= p["strings"] or not p["unit"]
    for h in (W.jw_hamiltonian(22, 96, 422), W.random_hamiltonian(22, 96, 322)):
        for p in plan_of(h, 0, sv.C64):
            assert not (p["unit"] and p["phases"])


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("dtype,n", [(sv.C64, 22), (sv.C128, 21)])
def test_values(dtype, n):
    rng = np.random.default_rng(n)
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dtype == sv.C64 else np.complex128)
    s = sv.StateVector(n, 0, dtype)
    s.set_state(psi)
    tol = 1e-5 if dtype == sv.C64 else 1e-12
    for h in few_cases(n) + pair_cases(n):
        ref = oracle.expect_terms(psi.astype(np.complex128), h).real
        assert np.max(np.abs(ref)) > 0
        _, pt = s.expect(h, sv.LAZY)
        assert np.max(np.abs(pt - ref)) < tol
        p, c = sv.hamiltonian_arrays(h)
        _, pt = sv.expect_noalloc(s.state, n, dtype, p, c)
        assert np.max(np.abs(pt - ref)) < tol
