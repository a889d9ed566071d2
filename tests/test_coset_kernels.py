"""Which kernel an expectation pass of few strings takes."""
import os
import subprocess

import numpy as np
import pytest

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
