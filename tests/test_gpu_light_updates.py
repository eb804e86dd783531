"""Renders without per-path records touch a path's radiance only where it
changes; the images hold the bits of the recorded paths' sums, for paths that
escape, emit, end at the depth limit or wait for a sun ray."""
import dataclasses

import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1912_04000_gb300.renderer import Renderer
    return Renderer(0)


@pytest.mark.parametrize("kw", [{}, {"bands_per_path": 4}, {"guided": True}])
@pytest.mark.parametrize("name,depth", [("prism_room", 1), ("prism_room", 7), ("tiny_box", 3), ("emissive", 5)])
def test_recorded_paths_sum_to_image(R, name, depth, kw):
    if name == "prism_room":
        wl = scenes.prism_room(width=19, height=13, n_bands=6, spp=3)
    else:
        wl = scenes.tiny_box(width=19, height=13, n_bands=6, spp=3)
    if name == "emissive":  # every wall glows a little
        mat = wl.scene.mat_type
        wl.scene = dataclasses.replace(wl.scene, mat_type=np.where(mat == scenes.LAMBERT, scenes.EMISSIVE, mat).astype(np.int32))
        le = np.broadcast_to(np.linspace(0.5, 1.5, 6, dtype=np.float32), wl.spectra.le.shape).copy()
        wl.spectra = dataclasses.replace(wl.spectra, le=le)
    R.load(wl)
    R.guide_init(seed=2, log2_table=10)
    plain = R.render(wl.cameras, 3, depth, 5, **kw)["spectral"].cpu().numpy()
    rec = R.render(wl.cameras, 3, depth, 5, probe_pixels=np.arange(19 * 13), **kw)
    L = rec["probe_L"].cpu().numpy().astype(np.float64).reshape(19 * 13, 3, 6)
    assert plain.any()
    assert np.array_equal(plain, rec["spectral"].cpu().numpy())
    assert np.array_equal(plain, (L[:, 0] + L[:, 1]) + L[:, 2])
