"""The default wave with little device memory free: an image that fits beside
the small wave's buffers, but not beside the large one's, is rendered."""
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


def test_image_that_leaves_room_for_the_small_wave_only():
    import torch

    from paper_1912_04000_gb300.renderer import Renderer

    # 192 bands of 3125 x 3125 pixels: 15.0 GB of spectral sums; the guided
    # waves' buffers take 1.5 GB (2^23 paths) and 3.0 GB (2^24)
    wl = scenes.tiny_box(width=3125, height=3125, n_bands=192, spp=1)
    R = Renderer(0).load(wl)
    R.guide_init(seed=1, log2_table=10)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = (16 << 30) + (300 << 20)
    held = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        out = R.render_host(wl.cameras, 1, 1, guided=1)
        assert out["stats"]["waves"] == -(-3125 * 3125 * 192 // (1 << 23))
        assert (out["xyz"] >= 0.0).all() and (out["xyz"] > 0.0).any()
    finally:
        del held
        R.close()
        torch.cuda.empty_cache()
