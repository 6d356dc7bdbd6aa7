"""The backward pass of dirac_apply takes the handle's own adjoint and force:
of any object with the handle's calls, of a subclass that replaces them, and of a handle on
which they were replaced (CPU test, with a stand-in for the library calls)."""
import pytest

torch = pytest.importorskip("torch")

from paper_1808_05506_gb300 import Dirac  # noqa: E402
from paper_1808_05506_gb300.autograd import dirac_apply  # noqa: E402


class Plain:
    """Only the calls that the differentiable apply makes of a handle."""

    def __init__(self):
        self.canon_dtype = torch.complex128
        self.links_generation = 0
        self.calls = []

    def set_links(self, V, remember=True):
        self.V = V.detach().clone()
        self.links_generation += 1

    def set_links_if_changed(self, V):
        self.set_links(V)
        return True

    def apply(self, x, out=None, dagger=False, layout=None):
        return x * self.V.sum()

    def apply_dagger(self, x, out=None, layout=None):
        self.calls.append("apply_dagger")
        return x * self.V.sum().conj()

    def force(self, psi, g, out=None):
        self.calls.append("force")
        return torch.full_like(self.V, (psi.conj() * g).sum())


def _loss(D):
    V = torch.randn(2, 2, 2, 2, 4, 3, 3, dtype=torch.complex128).requires_grad_(True)
    psi = torch.randn(2, 2, 2, 2, 1, 4, 3, dtype=torch.complex128).requires_grad_(True)
    dirac_apply(D, psi, V).abs().sum().backward()
    return psi.grad, V.grad


def test_any_object_with_the_calls():
    D = Plain()
    gpsi, gV = _loss(D)
    assert D.calls == ["apply_dagger", "force"] and gpsi is not None and gV is not None


def test_calls_replaced_on_one_handle():
    D = Dirac.__new__(Dirac)   # a handle without the library
    P = Plain()
    D.h = None
    D.canon_dtype, D.links_generation = P.canon_dtype, 0
    for name in ("set_links", "set_links_if_changed", "apply", "apply_dagger", "force"):
        setattr(D, name, getattr(P, name))
    gpsi, gV = _loss(D)
    assert P.calls == ["apply_dagger", "force"] and gpsi is not None and gV is not None


def test_backward_of_an_apply_that_a_wrapper_forwards():
    """A wrapper that forwards what it does not define keeps its own adjoint."""
    inner = Plain()

    class Wrapper:
        def __init__(self):
            self.calls = []

        def __getattr__(self, name):
            if name == "backward":   # the fused call of the handle inside
                return lambda psi, g: pytest.fail("the wrapper's own adjoint was passed by")
            return getattr(inner, name)

        def apply_dagger(self, x, out=None, layout=None):
            self.calls.append("apply_dagger")
            return inner.apply_dagger(x)

    D = Wrapper()
    _loss(D)
    assert D.calls == ["apply_dagger"] and inner.calls == ["apply_dagger", "force"]
