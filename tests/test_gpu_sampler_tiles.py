"""The tiled training pass against itself on fewer rows.  A row's outputs do
not depend on the rows beside it, and with dY in one row only every weight
gradient is one product and zeros, so both are equal bit for bit wherever the
row lies: in the first and last row of a tile, in a ragged last tile, and in
the second tile that a warpgroup works on (from 512 rows a multiprocessor)."""
import numpy as np
import pytest

from test_gpu_sampler import _setup, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,rows", [(129, [0, 127, 128]), (513, [511, 512]),
                                    (90001, [5, 77823, 77824, 89999, 90000])])
def test_a_row_does_not_depend_on_its_place(torch_cuda, B, rows):  # noqa: F811
    torch = torch_cuda
    _, s, _, _, Ut = _setup(torch, B)
    Y = s.forward(Ut).clone()
    for r in rows:
        # the same row alone among 128, in another place
        few = Ut[:128].clone()
        few[77] = Ut[r]
        assert torch.equal(s.forward(few)[77], Y[r])
        big, small = torch.zeros((B, 2), device="cuda"), torch.zeros((128, 2), device="cuda")
        big[r] = small[77] = torch.tensor([0.75, -1.25], device="cuda")
        assert np.array_equal(s.backward(Ut, big).cpu().numpy(), s.backward(few, small).cpu().numpy())
