"""The FP32 spectrum -> XYZ contraction at the edges of its stages (32 or 64
pixels, two to four in flight per CTA) and of its band counts (where the
stage size changes, one band, the largest), and with values outside the FP32
range, against the FP64 contraction."""
import numpy as np
import pytest

from paper_1912_04000_gb300 import _native, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1912_04000_gb300.renderer import Renderer
    return Renderer(0).load(scenes.tiny_box(n_bands=192, width=4, height=4))


@pytest.mark.parametrize("n_bands", [1, 7, 8, 16, 81, 105, 106, 107, 108, 192])
@pytest.mark.parametrize("n_pix", [1, 31, 32, 33, 63, 64, 65, 127, 64 * 304 + 1, 64 * 304 * 3 + 33])
def test_against_fp64(R, n_bands, n_pix):
    import torch
    if n_bands > 81 and n_pix > 64 * 304 + 1:
        n_pix = 32 * 304 * 3 + 17
    g = torch.Generator(device="cuda").manual_seed(n_pix * 200 + n_bands)
    s = torch.rand(n_pix, n_bands, device="cuda", dtype=torch.float64, generator=g) * 7.0
    s[torch.rand(s.shape, device="cuda", generator=g) < 0.1] = 0.0
    got = R.xyz(s, 192 - n_bands, 3, _native.XYZ_BF16X3).double()
    w = torch.from_numpy(scenes.tiny_box(n_bands=192, width=4, height=4).spectra.cmf_w).cuda().double()
    w = w[192 - n_bands:]
    want = s / 3.0 @ w
    # every product and sum in FP32: at most n / 8 + 8 roundings of 2^-24 on the sum of magnitudes
    bound = (n_bands / 8 + 8) * 2.0 ** -24 * (s / 3.0 @ w.abs()) + 1e-30
    assert bool(((got - want).abs() <= bound).all())


def test_values_outside_fp32(R):
    import torch
    s = torch.ones(70, 9, device="cuda", dtype=torch.float64)
    s[3, 2], s[40, 0], s[64, 8], s[65, 1], s[69, 5] = 1e300, float("inf"), float("nan"), 1e-300, 5e-324
    got = R.xyz(s, 80, 1, _native.XYZ_BF16X3).cpu().numpy()
    ref = R.xyz(s, 80, 1, _native.XYZ_FP64).cpu().numpy()
    plain = np.ones(70, bool)
    plain[[3, 40, 64]] = False
    np.testing.assert_allclose(got[plain], ref[plain], rtol=1e-6)
    assert not np.isfinite(got[[3, 40, 64]]).any(axis=1).all()
    assert np.isnan(got[64]).any() and not np.isfinite(got[3]).all() and not np.isfinite(got[40]).all()
