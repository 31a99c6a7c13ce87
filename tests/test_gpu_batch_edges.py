"""Batches, and batches without allocation, whose splats meet every edge of the windowed splat and of the map
choice table: views that cut the attractor, sizes down to one pixel, bounds
whose scaled upper end rounds to the size or below it, several thresholds in
one bucket, maps of probability 0.  Histograms and discards are whole numbers
and must equal the oracle's."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (view, W, H, channels)
VIEWS = [((0.0, 1.0, 0.0, 1.0), 64, 64, 4),          # the square fills it, edges included
         ((0.0, 1.0, 0.0, 1.0), 1, 1, 1),
         ((0.0, 1.0, 0.0, 1.0), 2, 3, 2),
         ((0.25, 0.75, -0.5, 0.3), 37, 23, 3),       # cuts through the attractor
         ((0.1, 0.7, 0.1, 0.9), 100, 333, 4),        # 1 / 0.6 and 1 / 0.8 are inexact
         ((1 / 3, 2 / 3, 1 / 7, 6 / 7), 49, 21, 16),
         ((-1e-3, 1.0, 0.0, 1.0 + 1e-6), 257, 255, 4),
         ((2.0, 3.0, 2.0, 3.0), 16, 16, 4)]          # nothing lands


def _systems():
    square = W.square_system()
    # thresholds 2^-9 apart share a bucket of the choice table (2^-7 wide),
    # and two maps are never chosen
    corners = [(0, 0), (1, 0), (0, 1), (1, 1), (0.5, 0.5), (0.25, 0.75), (0.75, 0.25)]
    many = W.System(2, [W.Map("affine", (0.5, 0.0, 0.0, 0.5, 0.5 * x, 0.5 * y)) for x, y in corners],
                    [1 / 512, 1 / 512, 0.0, 1 / 512, 0.4, 0.0, 0.6 - 3 / 512])
    # a map that throws points far out, to infinity and to NaN within a run
    wild = W.System(2, [W.Map("affine", (0.5, 0.0, 0.0, 0.5, 0.0, 0.0)),
                        W.Map("affine", (-1e20, 1e20, 1e20, 1e20, 1.0, 0.5))], [0.98, 0.02])
    return [square, many, wild]


@pytest.mark.parametrize("view", VIEWS)
@pytest.mark.parametrize("iters", [60, 61])
def test_batch_edges_equal_the_oracle(view, iters):
    torch = pytest.importorskip("torch")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    box, w, h, c = view
    d = W.Target("hist_u32", w, h, c, box)
    systems = _systems()
    n = [1, 700, 2049]
    tens = [cfs.alloc_target(d) for _ in systems]
    frames = [(cfs.System(s), m, 5 * j, j, [d], [t])
              for j, (s, m, t) in enumerate(zip(systems, n, tens))]
    b = cfs.Batch(cfs.Chain([W.Op("splat", (0,))], 2), frames, iters=iters, burn_in=20, seed=9)
    for ilp in (0, 1, 2):                        # the plan as created, then each program
        if ilp:
            b.set_plan(ilp=ilp, chunk=256)
        b.launch(clear=True)
        disc = b.discards()
        torch.cuda.synchronize()
        for j, s in enumerate(systems):
            ref = O.render(s, [W.Op("splat", (0,))], [d], n_points=n[j], iters=iters, burn_in=20,
                           seed=9, system_id=j, point_begin=5 * j)[0]
            got = tens[j].cpu().numpy().view(np.uint32)
            assert np.array_equal(got.reshape(ref.buf.shape), ref.buf), (j, ilp)
            assert int(got.sum()) + int(disc[j, 0]) == n[j] * (iters - 20), (j, ilp)


@pytest.mark.parametrize("view", VIEWS)
@pytest.mark.parametrize("iters,burn_in", [(60, 20), (41, 18), (23, 23), (3, 0)])
def test_noalloc_edges_equal_the_oracle(view, iters, burn_in):
    torch = pytest.importorskip("torch")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    box, w, h, c = view
    d = W.Target("hist_u32", w, h, c, box)
    # 51 frames (more than one launch's descriptors); frames 3 and up share one
    # small system, so that the oracle runs it once
    systems = _systems() + [W.sierpinski_system()] * 48
    n = [1, 700, 2049] + [65] * 48
    size = c * h * w
    # targets packed without gaps: most start on no 16-byte boundary
    flat = torch.full((size * len(systems) + 1,), 7, dtype=torch.int32, device="cuda")
    tens = [flat[1 + size * j:1 + size * (j + 1)].view(c, h, w) for j in range(len(systems))]
    frames = [(cfs.System(s), m, 5 * min(j, 3), min(j, 3), [d], [t])
              for j, (s, m, t) in enumerate(zip(systems, n, tens))]
    disc = torch.full((len(frames),), 9, dtype=torch.int64, device="cuda")
    for _ in range(2):
        cfs.render_batch_noalloc(frames, iters=iters, burn_in=burn_in, seed=9, discards=disc)
    torch.cuda.synchronize()
    assert int(flat[0]) == 7
    for j in range(len(frames)):
        if j <= 3:
            ref = O.render(systems[j], [W.Op("splat", (0,))], [d], n_points=n[j], iters=iters,
                           burn_in=burn_in, seed=9, system_id=j, point_begin=5 * j)[0].buf
        got = tens[j].cpu().numpy().view(np.uint32)
        assert np.array_equal(got.reshape(ref.shape), ref), j
        assert int(got.sum()) + int(disc[j]) == n[j] * (iters - burn_in), j
