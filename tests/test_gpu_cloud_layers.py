"""Stored clouds into layers around the size from which depth splats go without
reading first, and with more points than pixels: the layer is the same as from
the points in another order and in several calls, and bounds the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_02226_gb300 import workloads as W

from _parity import check_depth_close, fixed_margin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,n", [(8192, 1 << 20), (8192, 4), (4096, 1 << 20), (6144, 1 << 16),
                                 (64, 1 << 16)])
def test_layers_of_every_size(w, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    xyz, fn = cfs.pointcloud_generate(cfs.System(W.cloud_system()), n, 32, seed=2)
    t = W.cloud_target(w)
    ch = cfs.Chain(W.cloud_chain(21), 3)
    a, b = cfs.alloc_target(t), cfs.alloc_target(t)
    cfs.render_points(ch, xyz, fn, [t], [a])
    half = n // 2 // 4 * 4
    back = xyz.flip(1).contiguous(), fn.flip(0).contiguous()
    for lo, hi in ((half, n), (0, half)):
        if hi > lo:
            cfs.render_points(ch, back[0][:, lo:hi].contiguous(), back[1][lo:hi].contiguous(), [t], [b])
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    if n <= 1 << 16:
        o = O.render_points(np.ascontiguousarray(xyz.cpu().numpy().T), fn.cpu().numpy(),
                            W.cloud_chain(21), [t], margin_px=fixed_margin([t], 1e-5), track=True)[0]
        check_depth_close(a.cpu().numpy().view(np.uint64), o)
