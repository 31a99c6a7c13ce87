"""The cloud generator's map choice: 2^b equally likely maps (chosen by a
shift), other counts and nearly equal probabilities (chosen by comparisons),
maps of probability 0, and step counts on and off the four-step blocks.
Affine maps and indices are exact, so clouds equal the oracle's."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _probs():
    near = [0.125] * 8
    near[3] += 1e-9
    return [[1.0], [0.5, 0.5], [0.25] * 4, [3.0] * 8, [1 / 16] * 16, [1 / 3] * 3, near,
            [0.25, 0.25, 0.25, 0.25, 0.0], [0.0, 0.5, 0.5], [0.5, 0.0, 0.5, 0.0]]


@pytest.mark.parametrize("probs", _probs())
@pytest.mark.parametrize("dim", [2, 3])
def test_cloud_choice_equals_the_oracle(probs, dim):
    torch = pytest.importorskip("torch")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    rng = np.random.default_rng(len(probs))
    maps = [W.Map("affine", tuple(W.f32(v) for v in rng.uniform(-0.5, 0.5, 6 if dim == 2 else 12)))
            for _ in probs]
    s = W.System(dim, maps, probs)
    for n, iters in ((1, 1), (300, 3), (1025, 4), (700, 9), (257, 32)):
        xyz, fn = cfs.pointcloud_generate(cfs.System(s), n, iters, seed=11, system_id=3)
        torch.cuda.synchronize()
        ox, ofn = O.pointcloud_generate(s, n, iters, seed=11, system_id=3)
        assert np.array_equal(xyz.cpu().numpy().T, ox[:, :dim]), (n, iters)
        assert np.array_equal(fn.cpu().numpy(), ofn), (n, iters)
