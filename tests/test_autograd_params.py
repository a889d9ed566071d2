"""Parameter tensors that vqe_energy takes: any floating type, views and lazily
negated ones included.  The simulator is a stand-in (energy sum(p^2), gradient
2 p), so this runs without a GPU; the values are exact in every type."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
ag = pytest.importorskip("paper_2410_04252_gb300.autograd")


class Sim:
    def reset(self, index):
        self.index = index

    def grad(self, circ, params, ham=None, schedule=None, paulis=None, coeffs=None):
        assert isinstance(params, np.ndarray) and params.dtype == np.float64 and params.ndim == 1
        return float((params ** 2).sum()), 2.0 * params


VALUES = [0.5, -1.25, 2.0, 0.75]


def tensors():
    for dt in (torch.float64, torch.float32, torch.float16, torch.bfloat16):
        yield str(dt), torch.tensor(VALUES, dtype=dt)
    yield "strided", torch.tensor([v for v in VALUES for _ in range(2)], dtype=torch.float32)[::2]
    z = torch.complex(torch.zeros(4), -torch.tensor(VALUES))
    assert z.conj().imag.is_neg()
    yield "negated", z.conj().imag
    yield "negated64", z.to(torch.complex128).conj().imag


@pytest.mark.parametrize("name,p", list(tensors()), ids=lambda v: v if isinstance(v, str) else "")
@pytest.mark.parametrize("ham", [object(), (np.zeros((1, 2), np.uint64), np.ones(1))])
def test_parameter_types(name, p, ham):
    theta = p.detach().requires_grad_(True)
    e = ag.vqe_energy(theta, Sim(), None, ham)
    assert e.dtype == p.dtype and e.ndim == 0
    assert float(e) == sum(v * v for v in VALUES)
    e.backward()
    assert theta.grad.dtype == p.dtype
    assert theta.grad.tolist() == [2 * v for v in VALUES]
