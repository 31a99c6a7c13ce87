"""The tuner compares every batch's plan with the item sizes of the batch as
created, also with more shape classes than it tunes one by one, and takes no
older cache entry for an answer to that."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes", [2, 33])
def test_created_sizes_are_tried(classes, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_02226_gb300 import cfs
    descs = [W.animation_target(64 + j) for j in range(classes)]
    tens = [cfs.alloc_target(d) for d in descs]
    sys_ = cfs.System(W.square_system())
    frames = [(sys_, 2048, 0, j, [d], [t]) for j, (d, t) in enumerate(zip(descs, tens))]
    chain = cfs.Chain([W.Op("splat", (0,))], 2)
    path = tmp_path / "tune.txt"

    def tuned():
        b = cfs.Batch(chain, frames, iters=8, burn_in=4, seed=1)
        choice = b.tune()
        b.launch(clear=True)
        total = sum(int(t.sum()) for t in tens)
        assert total + int(np.asarray(b.discards()).sum()) == classes * 2048 * 4
        return choice

    cfs.tune_cache_clear()
    try:
        first = tuned()
        assert first["n_classes"] == classes
        # the program, each class where they are few, and the comparison
        assert cfs.tune_cache_size() == 2 + (classes if classes <= 32 else 0)
        assert tuned()["from_cache"]
        # a file of the time when the comparison left the created sizes out
        cfs.tune_cache_save(str(path))
        path.write_text("".join(line if line.split("|")[0] in ("batch", "class") else
                                line.replace(line.split("|")[0], "classes", 1)
                                for line in path.read_text().splitlines(True)))
        cfs.tune_cache_clear()
        cfs.tune_cache_load(str(path))
        again = tuned()
        assert not again["from_cache"] and 2 <= again["trials"] <= 3
    finally:
        cfs.tune_cache_clear()
