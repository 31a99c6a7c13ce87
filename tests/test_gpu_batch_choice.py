"""The map choice of batches, with and without allocation, around the edges of
its buckets (2^-5 and 2^-7 of the words): thresholds on a bucket's first and
last word, two in one bucket of either kind, 16 maps, a map that takes almost
everything.  Histograms are whole numbers and must equal the oracle's."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu

U = 2.0 ** -32
PROBS = {
    "one_map": [1.0],
    "first_word": [1 / 32, 1 / 2, 15 / 32],                      # T = 2^27: a bucket's first word
    "second_word": [1 / 32 + U, 1 / 2, 15 / 32 - U],
    "last_word": [1 / 32 - U, 1 / 2, 15 / 32 + U],
    "two_in_a_32nd": [1 / 64, 1 / 80, 0.3, 1.0 - 1 / 64 - 1 / 80 - 0.3],
    "two_in_a_128th": [1 / 256, 1 / 512, 0.5, 0.5 - 3 / 512],
    "sixteen": [1 / 16] * 16,
    "sixteen_uneven": [(j + 1) / 136 for j in range(16)],
    "almost_all": [U, 1.0 - 2 * U, U],
    "never": [0.0, 0.5, 0.0, 0.5, 0.0],
}


@pytest.mark.parametrize("name", sorted(PROBS))
def test_choice_at_bucket_edges(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    p = PROBS[name]
    maps = [W.Map("affine", (0.5, 0.1 * (j % 3), -0.1, 0.4, 0.05 * j, 0.6 - 0.03 * j))
            for j in range(len(p))]
    sysd = W.System(2, maps, p)
    d = W.Target("hist_u32", 96, 80, 16, (-1.0, 2.0, -1.0, 2.0))
    n, iters = 3001, 120
    ref = O.render(sysd, [W.Op("splat", (0,))], [d], n_points=n, iters=iters, burn_in=20, seed=5,
                   system_id=3, point_begin=11)[0].buf
    t = [cfs.alloc_target(d) for _ in range(2)]
    frames = [(cfs.System(sysd), n, 11, 3, [d], [x]) for x in t]
    b = cfs.Batch(cfs.Chain([W.Op("splat", (0,))], 2), frames[:1], iters=iters, burn_in=20, seed=5)
    for ilp in (0, 1, 2):                        # the plan as created, then each program
        if ilp:
            b.set_plan(ilp=ilp, chunk=256)
        b.launch(clear=True)
        torch.cuda.synchronize()
        got = t[0].cpu().numpy().view(np.uint32)
        assert np.array_equal(got.reshape(ref.shape), ref)
    cfs.render_batch_noalloc(frames[1:], iters=iters, burn_in=20, seed=5)
    torch.cuda.synchronize()
    assert torch.equal(t[0], t[1])
