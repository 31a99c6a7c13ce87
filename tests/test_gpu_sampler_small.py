"""Gradients of batches below one tile of 128 rows, on both sides of the 64 rows
from which their weight gradients take the row-major kernel, against the fp64
oracle on the same BF16-rounded operands."""
import numpy as np
import pytest

from oracle import sampler_oracle as SO

from test_gpu_sampler import _rel, _setup, _unflat, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [63, 64, 65, 127])
def test_small_batches_match_the_oracle(torch_cuda, B):  # noqa: F811
    torch = torch_cuda
    _, s, params, Ub, Ut = _setup(torch, B)
    dY = np.random.default_rng(B).normal(size=(B, 2)).astype(np.float32)
    g = s.backward(Ut, torch.from_numpy(dY).cuda()).cpu().numpy()
    _, cache = SO.forward(params, Ub, bf16=True)
    want = SO.backward(params, cache, dY, bf16=True)
    for l, (W_, b) in enumerate(_unflat(g)):
        assert _rel(W_, want[l][0]) < 2e-2 and _rel(b, want[l][1]) < 2e-2, l
