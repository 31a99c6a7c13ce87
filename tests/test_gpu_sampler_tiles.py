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


@pytest.mark.parametrize("B", [100, 4096])
def test_captured_step_replays_the_same(torch_cuda, B):  # noqa: F811
    # the backward's kernels start under each other's tails: their order holds in
    # a graph of the caller's too
    torch = torch_cuda
    cfs, s, _, _, Ut = _setup(torch, B)
    dY = torch.linspace(-1, 1, 2 * B, device="cuda").view(B, 2)
    Y, g = s.forward(Ut).clone(), s.backward(Ut, dY).clone()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        graph.capture_begin()
        Yc = s.forward(Ut, stream=stream)
        gc = s.backward(Ut, dY, stream=stream)
        graph.capture_end()
    for _ in range(3):
        gc.zero_()
        Yc.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(Yc, Y)
        assert float((gc - g).norm() / g.norm()) < 1e-5
