"""The sliced-Wasserstein kernel where its deal of sorts to warps can go wrong:
rounds that span several systems, groups without a sort, several rounds a CTA;
points that are not eight-byte aligned; equal points."""
import math

import numpy as np
import pytest

from oracle import sampler_oracle as SO

from test_gpu_sampler import _rel, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _points(S, N, P):
    rng = np.random.default_rng(S * N + P)
    X = rng.normal(size=(S, N, 2)).astype(np.float32)
    T = (rng.normal(size=(S, N, 2)) * 0.5 + 0.3).astype(np.float32)
    phi = (np.arange(P) * math.pi / P + 0.1).astype(np.float32)
    return X, T, phi


@pytest.mark.parametrize("S,N,P", [(1, 32, 1), (700, 32, 31), (5, 64, 33), (300, 64, 3),
                                   (7, 128, 9), (37, 256, 1), (9, 512, 65), (41, 1024, 21),
                                   (1300, 1024, 1)])
def test_deal_of_sorts(torch_cuda, S, N, P):  # noqa: F811
    torch = torch_cuda
    from paper_2606_02226_gb300 import cfs
    X, T, phi = _points(S, N, P)
    loss, dX = cfs.sw_loss(*(torch.from_numpy(a).cuda() for a in (X, T, phi)))
    Lo, go = SO.sw_loss_grad(X, T, phi.astype(np.float64))
    assert abs(float(loss.item()) - Lo) < 1e-5 * Lo
    assert _rel(dX.cpu().numpy(), go) < 1e-4


@pytest.mark.parametrize("off", [0, 1])
def test_points_of_any_alignment(torch_cuda, off):  # noqa: F811
    torch = torch_cuda
    from paper_2606_02226_gb300 import cfs
    X, T, phi = _points(3, 256, 5)

    def at(a, shift):
        flat = torch.zeros(a.size + 1, device="cuda")[shift:shift + a.size]
        return flat.copy_(torch.from_numpy(a).reshape(-1)).view(a.shape)

    p = torch.from_numpy(phi).cuda()
    want = cfs.sw_loss(at(X, 0), at(T, 0), p)
    got = cfs.sw_loss(at(X, off), at(T, 1 - off), p)
    # the same sorts and sums; only the order of the atomics differs
    assert abs(float(got[0].item()) - float(want[0].item())) < 1e-6 * float(want[0].item())
    assert _rel(got[1].cpu().numpy(), want[1].cpu().numpy()) < 1e-6


def test_equal_points_have_equal_gradients(torch_cuda):  # noqa: F811
    torch = torch_cuda
    from paper_2606_02226_gb300 import cfs
    X, T, phi = _points(2, 1024, 1)
    X[0, ::2] = X[0, 1::2]
    X[1, :] = 0.25
    _, dX = cfs.sw_loss(*(torch.from_numpy(a).cuda() for a in (X, T, phi)))
    g = dX.cpu().numpy()
    assert np.array_equal(g[0, ::2], g[0, 1::2]) and np.all(g[1] == g[1, 0])
