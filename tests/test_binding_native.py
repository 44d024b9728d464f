"""What the native half of the binding refuses before any call is made (no GPU needed), and that both halves drive one library."""
import pytest
import torch

from paper_1910_04732_b200 import binding as b
from paper_1910_04732_b200 import build


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


X = torch.zeros(4, 8, dtype=torch.bfloat16)


@pytest.mark.parametrize("bad,exc", [(X.t(), AssertionError), (X[0], AssertionError), (X[:, ::2], AssertionError), (X.half(), TypeError),
                                     (None, AttributeError), (3, TypeError)])
def test_matrices_of_another_form_are_refused(bad, exc):
    with pytest.raises(exc):
        b.compact_fwd(bad, X, X, X, 4, None)
    with pytest.raises(exc):
        b.gated_lowrank_bwd(X, bad, X, X, None, None, X, None, None, None, None, None)
    if bad is not None:
        with pytest.raises(exc):
            b.compact_ranks(torch.zeros(4), 0, (1.0, -0.1, 1.1), None, None, None, bad, X, X, X)


def test_every_native_call_has_its_python_name():
    native = b._native()
    names = [n for n in dir(native) if not n.startswith("_")]
    assert len(names) == 8 and all(callable(getattr(b, n)) and "flop_" + n in b.EXPORTS for n in names)
    with pytest.raises(TypeError):
        native.compact_fwd(X)
