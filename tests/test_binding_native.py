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


HC = (0.5, -0.25, 1.25)      # exact in every form


@pytest.mark.gpu
@pytest.mark.parametrize("hc", [list(HC), torch.tensor(HC), torch.tensor(HC).numpy(), dict(enumerate(HC)), [str(v) for v in HC]])
def test_constants_in_any_form_that_can_be_indexed(hc):
    la, z, want = torch.linspace(-3, 3, 64, device="cuda"), torch.zeros(64, device="cuda"), torch.zeros(64, device="cuda")
    b.gate_sample(la, HC, 1, 2, want)
    b.gate_sample(la, hc, 1, 2, z)
    assert torch.equal(z, want)


@pytest.mark.gpu
@pytest.mark.parametrize("accumulate,adds", [(False, False), (0, False), (0.5, False), ("0", False), (True, True), (2, True), (torch.tensor(1), True)])
def test_accumulate_is_an_integer(accumulate, adds):
    x = torch.ones(8, 8, device="cuda")
    v = torch.ones(8, device="cuda")
    dP, dQ, dla = 3 * x, 3 * x, 3 * v
    b.gated_lowrank_bwd(x, x, x, x, v, v, x, None, dP, dQ, dla, b.alloc_workspace(b.workspace_bytes(b.OP_BWD, 8, 8, 8, 8, b.F32)), accumulate)
    assert torch.all(dP == 8 + 3 * adds) and torch.all(dQ == 64 + 3 * adds) and torch.all(dla == 512 + 3 * adds)


def test_accumulate_that_is_no_integer_is_refused():
    with pytest.raises(TypeError):
        b.gated_lowrank_bwd(X, X, X, X, None, None, X, None, None, None, None, None, None)


def test_a_module_of_another_torch_is_not_loaded(monkeypatch):
    assert build.native_up_to_date()
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    monkeypatch.setattr(b, "_native_module", None)
    assert not build.native_up_to_date()
    with pytest.raises(RuntimeError, match="0.0.0"):
        b._native()
