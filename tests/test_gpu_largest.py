"""Renders and stored clouds of almost 2^32 points: every point once, the last
ones too."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOP = 1 << 32


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    return torch, cfs


@pytest.mark.parametrize("n", [TOP - 1, TOP - 4096])
def test_render_of_the_most_points(gpu, n):
    torch, cfs = gpu
    d = W.Target("hist_u32", 256, 256, 4, (0.0, 0.9, 0.0, 1.0))
    chain, sys_ = cfs.Chain([W.Op("splat", (0,))], 2), cfs.System(W.square_system())

    def render(parts):
        t = cfs.alloc_target(d)
        disc = torch.zeros(1, dtype=torch.int64, device="cuda")
        for begin, m in parts:
            cfs.render(sys_, chain, [d], [t], n_points=m, point_begin=begin, iters=1, burn_in=0,
                       seed=4, discards=disc)
        torch.cuda.synchronize()
        return t, int(disc)

    whole, disc = render([(0, n)])
    halves, want = render([(0, TOP // 2), (TOP // 2, n - TOP // 2)])
    assert torch.equal(whole, halves) and disc == want
    assert int((whole.to(torch.int64) & 0xFFFFFFFF).sum()) + disc == n


def test_cloud_of_the_most_points(gpu):
    torch, cfs = gpu
    n = TOP - 3
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    from oracle import oracle as O
    sys_ = W.sierpinski_system()
    xyz, fn = cfs.pointcloud_generate(cfs.System(sys_), n, iters=2, seed=7)
    torch.cuda.synchronize()
    # the cloud's point i does not depend on how many there are
    for first in (0, TOP // 2 - 5, n - 1000):
        ids = np.arange(first, first + 1000, dtype=np.uint64).astype(np.uint32)
        k, p, _ = O.trace(sys_, [], ids, iters=2, seed=7)
        assert np.array_equal(fn[first:first + 1000].cpu().numpy(), k[:, -1])
        assert np.array_equal(xyz[:, first:first + 1000].cpu().numpy().T, p[:, -1, :2])
