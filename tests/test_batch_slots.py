"""Batches whose chain splats into another target than the first: no privatized
window, which belongs to target 0, and the oracle's histograms."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W


def _targets(slot):
    return [W.Target("hist_u32", 40 + 8 * j, 50, 1 + j, (-0.1, 1.1, -0.1, 1.1))
            for j in range(slot + 1)]


@pytest.mark.parametrize("slot", [0, 1, 3])
def test_only_target_0_has_a_window(slot):
    from paper_2606_02226_gb300 import cfs
    src, _ = cfs.codegen_check(cfs.System(W.square_system()), cfs.Chain([W.Op("splat", (slot,))], 2),
                               _targets(slot), mode=2)
    assert ("#define CFS_TILE 1" in src) == (slot == 0)
    assert ("cfs_splat_hist_tile" in src) == (slot == 0)


@pytest.mark.gpu
@pytest.mark.parametrize("slot", [1, 3])
@pytest.mark.parametrize("ilp", [1, 2])
def test_splats_into_another_target(slot, ilp):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    descs, ops = _targets(slot), [W.Op("splat", (slot,))]
    systems, n = [W.square_system(), W.sierpinski_system()], [3001, 70]
    tens = [[cfs.alloc_target(d) for d in descs] for _ in systems]
    frames = [(cfs.System(s), m, 5 * j, j, descs, t)
              for j, (s, m, t) in enumerate(zip(systems, n, tens))]
    b = cfs.Batch(cfs.Chain(ops, 2), frames, iters=41, burn_in=20, seed=9)
    b.set_plan(ilp=ilp)
    b.launch(clear=True)
    disc = np.asarray(b.discards())
    for j, s in enumerate(systems):
        ref = O.render(s, ops, descs, n_points=n[j], iters=41, burn_in=20, seed=9, system_id=j,
                       point_begin=5 * j)
        for t in range(slot + 1):
            got = tens[j][t].cpu().numpy().view(np.uint32)
            assert np.array_equal(got.reshape(ref[t].buf.shape), ref[t].buf), (j, t)
        assert int(got.sum()) + int(disc[j, slot]) == 21 * n[j]
    assert (b.windows()[..., 2] < 0).all()
