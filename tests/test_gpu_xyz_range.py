"""Spectral sums whose weighted sum is above the FP32 range while the image
(that sum over the samples) is within it, and sums above the range
themselves."""
import dataclasses

import pytest

from paper_1912_04000_gb300 import _native, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bands", [1, 16, 81, 192])
def test_large_sums_of_many_samples(n_bands):
    import torch

    from paper_1912_04000_gb300.renderer import Renderer

    spp, n_pix = 100_000, 64 * 304 + 37
    wl = scenes.tiny_box(n_bands=192, width=4, height=4)
    R = Renderer(0).load(dataclasses.replace(
        wl, spectra=dataclasses.replace(wl.spectra, cmf_w=wl.spectra.cmf_w * 683.0)))
    g = torch.Generator(device="cuda").manual_seed(n_bands)
    # sums of 2^90 .. 2^134, a few of ordinary size among them
    s = torch.exp2(90.0 + 44.0 * torch.rand(n_pix, 1, device="cuda", dtype=torch.float64, generator=g))
    s = s * torch.rand(n_pix, n_bands, device="cuda", dtype=torch.float64, generator=g)
    s[::7] *= 2.0 ** -100
    got = R.xyz(s, 192 - n_bands, spp, _native.XYZ_BF16X3).double()
    w = torch.from_numpy(wl.spectra.cmf_w * 683.0).cuda().double()[192 - n_bands:]
    want, mag = s / spp @ w, s / spp @ w.abs()
    assert float(mag.max()) < 3e38
    # every product and sum in FP32: at most n / 8 + 8 roundings of 2^-24 on the sum of magnitudes
    bound = (n_bands / 8 + 8) * 2.0 ** -24 * mag + 1e-30
    assert bool(((got - want).abs() <= bound).all())
