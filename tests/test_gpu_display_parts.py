"""The display where a layer of few pixels is dealt to several CTAs an item:
sizes at the edges of a part (1024 pixels and up) and of an item (8192)."""
import pytest

from test_gpu_display import _run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["hist_u32", "rgba_f32", "depth_u64"])
@pytest.mark.parametrize("Wd,H", [(1, 1), (1023, 1), (1024, 1), (1025, 1), (8191, 1), (8196, 1),
                                  (320, 240), (1217, 1024), (2432, 2048), (2049, 2432)])
def test_parts_of_items(torch_cuda, kind, Wd, H):  # noqa: F811
    n_diff, o = _run(torch_cuda, kind, Wd, H, seed=Wd + H, gamma=2.2, background=0x01020304)
    assert n_diff <= max(1, 1e-3 * o.size)
