"""Waves of several whole samples: the same bits as one sample (or less) per
wave, for one and four bands, guided paths, progressive accumulation, sample
counts that leave a remainder, and per-path records."""
import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1912_04000_gb300.renderer import Renderer
    r = Renderer(0)
    r.wl = scenes.prism_room(width=23, height=17, n_bands=11, spp=1, depth=6)
    r.load(r.wl)
    r.guide_init(seed=3, log2_table=12)
    return r


@pytest.mark.parametrize("kw", [{}, {"bands_per_path": 4}, {"guided": True}])
@pytest.mark.parametrize("spp,fit", [(2, 2), (5, 2), (7, 3), (4, 64)])
def test_samples_per_wave(R, kw, spp, fit):
    wl = R.wl
    units = (11 + 3) // 4 if kw.get("bands_per_path") == 4 else 11
    per_sample = 23 * 17 * units
    probe = [0, 7, 390]
    one = R.render(wl.cameras, spp, wl.depth, 9, wave_capacity=per_sample, probe_pixels=probe, **kw)
    part = R.render(wl.cameras, spp, wl.depth, 9, wave_capacity=per_sample - 5, **kw)
    many = R.render(wl.cameras, spp, wl.depth, 9, wave_capacity=fit * per_sample + 3, probe_pixels=probe, **kw)
    assert many["stats"]["waves"] == -(-spp // min(fit, spp)) and one["stats"]["waves"] == spp
    for key in ("spectral", "probe_L", "probe_sig"):
        assert np.array_equal(many[key].cpu().numpy(), one[key].cpu().numpy()), key
    assert np.array_equal(part["spectral"].cpu().numpy(), one["spectral"].cpu().numpy())


def test_progressive_samples(R):
    wl = R.wl
    whole = R.render(wl.cameras, 9, wl.depth, 4)["spectral"]
    out = R.render(wl.cameras, 4, wl.depth, 4)["spectral"]
    out = R.render(wl.cameras, 5, wl.depth, 4, sample_first=4, accumulate=True, out_spectral=out)["spectral"]
    assert np.array_equal(out.cpu().numpy(), whole.cpu().numpy())


def test_photon_camera_samples(R):
    wl = R.wl
    a = R.render_photons(wl.cameras, 5, wl.depth, 2, n_photons=2048)["spectral"].cpu().numpy()
    parts = [R.render_photons(wl.cameras, 5, wl.depth, 2, n_photons=2048, band_first=b, band_count=1)["spectral"]
             .cpu().numpy() for b in range(11)]
    np.testing.assert_allclose(np.concatenate(parts, 1), a, rtol=1e-6, atol=1e-12)
