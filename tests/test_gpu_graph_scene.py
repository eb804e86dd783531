"""Captured renders after the scene, the spectra or the guide were set again,
in tables of the same sizes: the image is that of the new scene, bit for bit
the one of a render without capture."""
import dataclasses

import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("change", ["sun", "scene", "guide"])
def test_replay_after_the_scene_changed(change):
    import torch

    from paper_1912_04000_gb300.renderer import Renderer

    wl = scenes.prism_room(width=64, height=48, n_bands=16)
    R = Renderer(0).load(wl, builder=1)
    guided = change == "guide"
    if guided:
        R.guide_init(seed=1, log2_table=12, n_min=4.0, n_max=64.0)
    out = {"out_spectral": torch.empty((wl.n_pixels, 16), dtype=torch.float64, device="cuda"),
           "out_xyz": torch.empty((wl.n_pixels, 3), dtype=torch.float32, device="cuda")}

    def render(use_graph):
        R.render(wl.cameras, 2, wl.depth, 3, use_graph=use_graph, guided=guided, **out)
        return [o.clone() for o in out.values()]

    before = render(True)
    assert all(torch.equal(a, b) for a, b in zip(before, render(False)))
    if change == "sun":
        sun = scenes.sun_direction(55.0, 190.0)
        R.set_spectra(dataclasses.replace(wl.spectra, sun_dir=sun, sun_half_angle=0.1))
    elif change == "scene":
        verts = wl.scene.verts.copy()
        verts[:, 0] *= 1.25
        R.load(dataclasses.replace(wl, scene=dataclasses.replace(wl.scene, verts=verts)), builder=1)
    else:
        R.guide_init(seed=1, log2_table=12, n_min=8.0, n_max=256.0)
    after = render(True)
    assert all(torch.equal(a, b) for a, b in zip(after, render(False)))
    assert not torch.equal(after[0], before[0])
