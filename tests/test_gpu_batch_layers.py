"""Item sizes as created: no larger than keeps the layers of the frames at work
in half of the L2, and, without a window, 4096 points where fewer would bring
fewer frames to work, larger ones where the layers are small, smaller ones where
CTAs would have no work -- and the same picture as with any other size."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _batch(cfs, kind, w, n, frames, iters=4):
    d = W.Target(kind, w, w, 1, (-1.0, 1.0, -1.0, 1.0), palette=W.palette_rgba(4),
                 palette8=W.palette_rgba8(8))
    ops, dim, sys_ = [W.Op("splat", (0,))], 2, W.square_system()
    if kind == "depth_u64":
        sys_, dim = W.cloud_system(), 3
        ops = [W.Op("translate3", (0.0, 0.0, 8.0)), W.Op("perspective", (3.5, 1e-3))] + ops
    tens = [cfs.alloc_target(d) for _ in range(frames)]
    s = cfs.System(sys_)
    b = cfs.Batch(cfs.Chain(ops, dim), [(s, n, 0, j, [d], [t]) for j, t in enumerate(tens)],
                  iters=iters, burn_in=1, seed=1)
    return b, tens


@pytest.mark.parametrize("kind,w,n,frames,sizes", [
    ("rgba_f32", 2048, 1 << 20, 8, "4096"),              # two layers are more than L2
    ("rgba_f32", 64, 1 << 18, 64, "larger"),
    ("rgba_f32", 64, 1 << 18, 8, "4096"),                # 512 items of 4096 on 304 CTAs
    ("rgba_f32", 64, 1 << 14, 4, "smaller"),
    ("depth_u64", 64, 1 << 18, 8, "smaller")])
def test_sizes_of_windowless_batches(kind, w, n, frames, sizes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    b, tens = _batch(cfs, kind, w, n, frames)
    info = b.info()
    if not 256 <= torch.cuda.get_device_properties(0).multi_processor_count * 2 <= 512:
        pytest.skip("sizes stated for 128 to 256 multiprocessors")
    plain = frames * -(-n // 4096)
    assert {"4096": info["n_items"] == plain, "larger": info["n_items"] < plain,
            "smaller": info["n_items"] > plain}[sizes], (info, plain)
    b.launch(clear=True)
    got, disc = [t.clone() for t in tens], np.asarray(b.discards()).copy()
    b.set_plan(chunk=4096)
    b.launch(clear=True)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(got, tens))
    assert np.array_equal(disc, np.asarray(b.discards()))


@pytest.mark.parametrize("w,most", [(2048, 16384), (256, 65536)])
def test_windowed_layers_stay_in_l2(w, most):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    n, frames = 1 << 20, 32
    d = W.Target("hist_u32", w, w, 4, (0.0, 1.0, 0.0, 1.0))
    tens = [cfs.alloc_target(d) for _ in range(frames)]
    s = cfs.System(W.square_system())
    b = cfs.Batch(cfs.Chain([W.Op("splat", (0,))], 2),
                  [(s, n, 0, j, [d], [t]) for j, t in enumerate(tens)], iters=4, burn_in=1, seed=1)
    grid = b.info()["grid"]
    if grid != 152 or not 120e6 < torch.cuda.get_device_properties(0).L2_cache_size < 140e6:
        pytest.skip("sizes stated for 152 multiprocessors and 126 MB of L2")
    want = 0
    for f in range(frames):
        share = (frames - 1 - f) * n // (4 * grid) // 2048 * 2048
        want += -(-n // max(4096, min(most, share)))
    assert b.info()["n_items"] == want
    b.launch(clear=True)
    assert sum(int(t.view(torch.int32).sum()) for t in tens) + int(np.asarray(b.discards()).sum()) \
        == frames * n * 3
