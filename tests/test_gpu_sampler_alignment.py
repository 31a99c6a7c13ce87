"""Gradients of the outputs that start on any four-byte boundary: a view at an
odd offset gives the weight gradients of an aligned copy, in batches below and
above one tile of rows."""
import pytest

from test_gpu_sampler import _setup, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 100, 128, 1000])
def test_backward_takes_any_alignment(torch_cuda, B):  # noqa: F811
    torch = torch_cuda
    _, s, _, _, Ut = _setup(torch, B)
    flat = torch.linspace(-1, 1, 2 * B + 1, device="cuda")
    view = flat[1:].view(B, 2)
    assert view.is_contiguous() and view.data_ptr() % 8 == 4
    want, got = s.backward(Ut, view.clone()), s.backward(Ut, view)
    # the same products and sums; only the order of the atomics differs
    assert float((got - want).norm() / want.norm()) < 1e-5
