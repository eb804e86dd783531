"""The default wave size: renders of more than 2^23 paths run in waves of up
to 2^24 with the same bits as in waves of 2^23; waves that keep guide training
records stay at 2^23 paths."""
import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1912_04000_gb300.renderer import Renderer
    r = Renderer(0)
    r.wl = scenes.prism_room(width=480, height=256, n_bands=72, spp=1, depth=4)  # 8.8 million paths per sample
    r.load(r.wl)
    r.guide_init(seed=3, log2_table=12)
    return r


@pytest.mark.parametrize("kw,small,large", [({}, 2, 1), ({"guided": True}, 2, 1), ({"bands_per_path": 4}, 1, 1)])
def test_same_bits(R, kw, small, large):
    a = R.render(R.wl.cameras, 1, 4, 9, wave_capacity=1 << 23, **kw)
    b = R.render(R.wl.cameras, 1, 4, 9, **kw)
    if R.torch.cuda.mem_get_info()[0] >= 20 << 30:
        assert (a["stats"]["waves"], b["stats"]["waves"]) == (small, large)
    assert np.array_equal(a["spectral"].cpu().numpy(), b["spectral"].cpu().numpy())


def test_training_waves(R):
    st = R.render(R.wl.cameras, 1, 4, 9, guided=True, guide_collect=64)["stats"]
    assert st["waves"] == 2
