"""Argument marshalling of the short calls: what is no dense tensor is a Python error (no GPU needed: the context is null)."""
import numpy as np
import pytest
import torch

F = torch.zeros(4, 16)


def _accept_scan(x0):
    from paper_2411_11925_b200 import _marshal, api  # noqa: F401  (api hands _marshal its address function)
    return _marshal.accept_scan(0, 1, 4, 16, 0.0, 1.0, 1.0, x0, F, F, F, F, torch.zeros(4, dtype=torch.int32), None)


def test_dense_tensors_and_arrays_reach_the_library():
    assert _accept_scan(F) == -1 and _accept_scan(np.zeros((4, 16), np.float32)) == -1 and _accept_scan(None) == -1   # null context


@pytest.mark.parametrize("make,error", [
    (lambda: F.t(), AssertionError),
    (lambda: F.to_sparse(), (AssertionError, RuntimeError)),
    (lambda: [0.0], TypeError),
])
def test_other_layouts_raise(make, error):
    with pytest.raises(error):
        _accept_scan(make())


def test_batched_tensors_raise():
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda t: torch.tensor(_accept_scan(t)))(torch.zeros(2, 4, 16))


def test_mixtures_without_a_component_axis_raise():
    from paper_2411_11925_b200 import _marshal, api  # noqa: F401
    ragged = torch.nested.nested_tensor([torch.zeros(2), torch.zeros(3)])
    for logw, error in ((ragged, RuntimeError), (torch.zeros(4), IndexError)):
        with pytest.raises(error):
            _marshal.gmm_draft_sample(0, 1, 4, (logw, F, F), F, F, F, None)
    with pytest.raises(ValueError):
        _marshal.gmm_draft_sample(0, 1, 4, (F, F), F, F, F, None)
