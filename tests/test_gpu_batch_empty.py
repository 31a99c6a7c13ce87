"""Frames without points between, before and after others: they get no items,
their histograms stay zero and the other frames are the oracle's."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [[3000, 0, 77, 0], [0, 1, 0, 0, 2049], [0, 0]])
@pytest.mark.parametrize("chunk", [0, 256])
def test_frames_of_no_points(n, chunk):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    fr = W.animation_frames(n_frames=len(n), seed=2)
    d = W.animation_target(64)
    ops = [W.Op("splat", (0,))]
    tens = [cfs.alloc_target(d) for _ in n]
    for t in tens:
        t.fill_(7)
    frames = [(cfs.System(f.system), m, 3 * j, j, [d], [t])
              for j, (f, m, t) in enumerate(zip(fr, n, tens))]
    b = cfs.Batch(cfs.Chain(ops, 2), frames, iters=26, burn_in=20, seed=4)
    if chunk:
        b.set_plan(chunk=chunk)
    b.launch(clear=True)
    disc = np.asarray(b.discards()).reshape(len(n), -1)[:, 0]
    for j, (f, m) in enumerate(zip(fr, n)):
        got = tens[j].cpu().numpy().view(np.uint32)
        assert int(got.sum()) + int(disc[j]) == 6 * m
        if m:
            ref = O.render(f.system, ops, [d], n_points=m, iters=26, burn_in=20, seed=4,
                           system_id=j, point_begin=3 * j)[0].buf
            assert np.array_equal(got.reshape(ref.shape), ref), j
