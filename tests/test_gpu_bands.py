"""The band texture's colour index at the edges of its modulo: every band
count, negative and huge band numbers, the guarded range |t| < 1e9 and beyond.
The square's coordinates and the band argument are exact FP32 operations, so
histograms over the colour index equal the oracle's."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", list(range(1, 17)))
def test_band_colours_equal_the_oracle(n):
    torch = pytest.importorskip("torch")
    from oracle import oracle as O
    from paper_2606_02226_gb300 import cfs
    d = W.Target("hist_u32", 4, 4, 16, (0.0, 1.0, 0.0, 1.0))
    s = W.square_system()
    for freq, phase in ((3.0, 0.5), (-7.0, 0.25), (1000.0, -512.0), (-9.99e8, 0.0), (2e9, -1e9),
                        (1e20, 1.0)):
        ops = [W.Op("bands", (1.0, freq, phase, float(n), float(16 - n))), W.Op("splat", (0,))]
        t = cfs.alloc_target(d)
        cfs.render(cfs.System(s), cfs.Chain(ops, 2), [d], [t], n_points=700, iters=60, burn_in=20,
                   seed=4)
        torch.cuda.synchronize()
        ref = O.render(s, ops, [d], n_points=700, iters=60, burn_in=20, seed=4)[0].buf
        assert np.array_equal(t.cpu().numpy().view(np.uint32).reshape(ref.shape), ref), (freq, phase)
