"""Palettes of every shape that a target may carry: rows past the sixteenth and
columns past the fourth are left out, an empty one sets nothing, any other
shape is an error -- and nothing beyond the palette's own field is written."""
import numpy as np
import pytest

from paper_2606_02226_gb300 import workloads as W

GREY = np.arange(24, dtype=np.float32)


def _target(palette=None, palette8=None):
    from paper_2606_02226_gb300 import cfs
    d = W.Target("rgba_f32", 8, 8, 1, (0.0, 1.0, 0.0, 1.0))
    object.__setattr__(d, "palette", palette)
    object.__setattr__(d, "palette8", palette8)
    plain = W.Target("rgba_f32", 8, 8, 1, (0.0, 1.0, 0.0, 1.0))
    object.__setattr__(plain, "palette", None)
    object.__setattr__(plain, "palette8", None)
    arr, _ = cfs.make_targets([d, plain], None, fake_ptr=True)
    want, _ = cfs.make_targets([plain, plain], None, fake_ptr=True)
    got, ref = bytearray(bytes(arr)), bytes(want)
    for field in (cfs.cfs_target.palette, cfs.cfs_target.palette8):
        if (palette is None) == (field is cfs.cfs_target.palette):
            continue
        got[field.offset:field.offset + field.size] = ref[field.offset:field.offset + field.size]
    assert bytes(got) == ref                 # all but the palette itself
    t = arr[0]
    return (np.array([[t.palette[k][c] for c in range(4)] for k in range(16)], np.float32),
            np.array(list(t.palette8), np.uint32))


@pytest.mark.parametrize("p,rows", [(GREY.reshape(6, 4), 6), (GREY.reshape(4, 6), 4),
                                    (GREY.reshape(4, 6).T, 6), ([[1, 2, 3, 4]], 1),
                                    (np.ones((20, 4)), 16), ([], 0), (np.zeros((0, 4)), 0),
                                    (np.zeros((0, 3)), 0)])
def test_palette(p, rows):
    got, _ = _target(palette=p)
    if rows:
        assert np.array_equal(got[:rows], np.asarray(p, np.float32)[:rows, :4])
    assert not got[rows:].any()


@pytest.mark.parametrize("p,rows", [([1, 2, 3], 3), (np.arange(1, 21), 16), ([], 0),
                                    (np.zeros((0, 2)), 0)])
def test_packed_palette(p, rows):
    _, got = _target(palette8=p)
    assert np.array_equal(got[:rows], np.asarray(p, np.uint32)[:rows].reshape(rows))
    assert not got[rows:].any()


@pytest.mark.parametrize("p,error", [(GREY, IndexError), (3.0, IndexError),
                                     (GREY.reshape(8, 3), IndexError),
                                     (GREY.reshape(6, 4, 1), TypeError),
                                     (GREY.reshape(3, 4, 2), TypeError),
                                     (np.zeros((2, 4, 0)), TypeError)])
def test_palette_refused(p, error):
    with pytest.raises(error):
        _target(palette=p)


@pytest.mark.parametrize("p,error", [(5, IndexError), (np.ones((2, 1)), TypeError),
                                     (np.ones((16, 9)), TypeError)])
def test_packed_palette_refused(p, error):
    with pytest.raises(error):
        _target(palette8=p)
