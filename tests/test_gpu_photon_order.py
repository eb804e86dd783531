"""Path orders and ray classes that depend on the call: the photon camera pass
walks runs of eight pixels of one band, so images whose last run is short are
compared with one-band renders (whose order is the pixel order); camera rays
use the box test for origins inside the scene bounds only where every camera
lies there."""
import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1912_04000_gb300.renderer import Renderer
    return Renderer(0)


@pytest.mark.parametrize("size", [(1, 1), (7, 1), (8, 1), (3, 3), (17, 5)])
def test_pixel_runs(R, size):
    wl = scenes.tiny_box(width=size[0], height=size[1], n_bands=5, spp=2, depth=5)
    R.load(wl)
    kw = dict(n_photons=2048, photon_depth=4, r_global=0.15, xyz_mode=2)
    a = R.render_photons(wl.cameras, 2, 5, 3, **kw)["spectral"].cpu().numpy()
    assert a.shape[0] == size[0] * size[1] and (a > 0).any()
    for b in range(5):
        one = R.render_photons(wl.cameras, 2, 5, 3, band_first=b, band_count=1, **kw)["spectral"].cpu().numpy()
        # the same FP32 path values, at most three FP64 additions in another order
        np.testing.assert_allclose(a[:, b], one[:, 0], rtol=1e-6, atol=1e-12)


def test_cameras_inside_and_outside(R):
    wl = scenes.prism_room(width=37, height=23, n_bands=3, spp=2)
    R.load(wl)
    c = wl.cameras[0]
    lo, hi = wl.scene.verts.min(0), wl.scene.verts.max(0)
    out = scenes.Camera(tuple(hi + 0.7 * (hi - lo)), tuple(0.5 * (lo + hi)), c.up, 50.0, 37, 23)
    axis = scenes.Camera(c.pos, (c.pos[0], c.pos[1], c.pos[2] + 1.0), (0.0, 1.0, 0.0), 50.0, 37, 23)  # rays with zero components
    n = 37 * 23
    alone = R.render([c, axis], 2, wl.depth, 5, xyz_mode=2)["spectral"].cpu().numpy()
    both = R.render([c, axis, out], 2, wl.depth, 5, xyz_mode=2)["spectral"].cpu().numpy()
    assert alone.shape[0] == 2 * n and both.shape[0] == 3 * n
    # both box tests admit every triangle that is hit: the same closest hits.
    # (Paths are numbered through the views: the first sample of a batch's
    # leading views keeps its random numbers, so the bits agree.)
    assert np.array_equal(alone, both[:2 * n])
