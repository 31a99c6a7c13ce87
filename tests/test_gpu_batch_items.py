"""A batch as created cuts its frames into items of falling sizes: frames of
many items of 65536 points, of one short item, and of none, equal to the same
frames in items of one size."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [[40_000_000, 1, 123_457, 0, 65_537, 2047], [3_000_001, 2_000_000],
                               [5_000_000] * 4 + [33]])
def test_created_items_equal_items_of_one_size(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    fr = W.animation_frames(n_frames=len(n), seed=2)
    d = W.animation_target(256)
    tens = [cfs.alloc_target(d) for _ in n]
    frames = [(cfs.System(f.system), m, 3 * j, j, [d], [t])
              for j, (f, m, t) in enumerate(zip(fr, n, tens)) if m > 0]
    b = cfs.Batch(cfs.Chain([W.Op("splat", (0,))], 2), frames, iters=26, burn_in=20, seed=4)
    got = []
    for chunk in (0, 4096):                      # as created, then items of 4096
        if chunk:
            b.set_plan(chunk=chunk)
        b.launch(clear=True)
        disc = np.asarray(b.discards())
        got.append(([t.cpu().numpy().copy() for f in frames for t in f[5]], disc))
    for x, y in zip(got[0][0], got[1][0]):
        assert np.array_equal(x, y) and x.any()
    assert np.array_equal(got[0][1], got[1][1])
    assert sum(int(x.view(np.uint32).sum(dtype=np.uint64)) for x in got[0][0]) + \
        int(got[0][1].sum()) == 6 * sum(n)
