"""Batch frames of almost 2^32 points, whose last item ends beside the end of
the 32-bit point range.  Every point counts: the frame's histogram is the sum
of its two halves' (the same points through ``point_begin``), and splats and
discards together are its points."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOP = 1 << 32


@pytest.mark.parametrize("n,plan", [
    (TOP - 8192, {}),
    (TOP - 8192, {"ilp": 1}),
    (TOP - 8192, {"chunk": 65536}),                  # the largest items of a batch as created
    (TOP - 8192, {"chunk": 1 << 20}),
    (TOP - 1, {"chunk": 4096}),
    (TOP - 32, {"chunk": 32 * 511, "ilp": 2}),       # items that end on n itself
    (TOP - 32, {"chunk": 32 * 511, "ilp": 1})])
def test_every_point_of_the_largest_frames(n, plan):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    d = W.Target("hist_u32", 256, 256, 4, (0.0, 0.9, 0.0, 1.0))
    chain, sys_ = cfs.Chain([W.Op("splat", (0,))], 2), cfs.System(W.square_system())

    def batch(parts, plan):
        tens = [cfs.alloc_target(d) for _ in parts]
        frames = [(sys_, m, begin, 3, [d], [t]) for (begin, m), t in zip(parts, tens)]
        b = cfs.Batch(chain, frames, iters=1, burn_in=0, seed=4)
        if plan:
            b.set_plan(**plan)
        b.launch(clear=True)
        disc = int(np.asarray(b.discards()).sum())
        return sum(t.cpu().numpy().view(np.uint32).astype(np.uint64) for t in tens), disc

    half = TOP // 2
    want, want_disc = batch([(0, half), (half, n - half)], {"chunk": 4096})
    assert int(want.sum()) + want_disc == n
    got, disc = batch([(0, n)], plan)
    assert int(got.sum()) + disc == n
    assert disc == want_disc and np.array_equal(got, want)
