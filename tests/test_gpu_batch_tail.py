"""Item sizes of a batch as created: the last large frame is cut as finely as
it would be alone, in items of 4096 points from 16384 points a CTA on, so that
no CTA waits for one long last item; frames before it may have larger ones."""
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [[1 << 22], [12_000_000], [1 << 16, 1 << 22], [1 << 24, 1 << 22]])
def test_the_last_frame_is_cut_finely(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    d = W.animation_target(128)
    tens = [cfs.alloc_target(d) for _ in n]
    sys_ = cfs.System(W.square_system())
    frames = [(sys_, m, 0, j, [d], [t]) for j, (m, t) in enumerate(zip(n, tens))]
    b = cfs.Batch(cfs.Chain([W.Op("splat", (0,))], 2), frames, iters=4, burn_in=0, seed=1)
    grid, items = b.info()["grid"], b.info()["n_items"]
    if sum(n) < 16384 * grid:
        pytest.skip("made for GPUs of up to 256 multiprocessors")
    last = -(-n[-1] // 4096)
    if len(n) == 1:
        assert items == last
    else:                                    # larger items in the frames before it
        assert last < items < last + -(-n[0] // 4096)
