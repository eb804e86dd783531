"""A captured render after other renders on the same context have replaced
buffers that it was captured with: the next replay gives the bits of the
first."""
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("between", ["more_samples", "larger_image"])
@pytest.mark.parametrize("kind", ["four_bands", "guided"])
def test_replay_after_buffers_grew(kind, between):
    import torch

    from paper_1912_04000_gb300.renderer import Renderer

    wl = scenes.prism_room(width=64, height=48, n_bands=16)
    big = scenes.prism_room(width=160, height=120, n_bands=16)
    R = Renderer(0).load(wl)
    R.guide_init(seed=1, log2_table=12)
    opts = {"bands_per_path": 4} if kind == "four_bands" else {"guided": True}
    # the queues of one-band paths are large enough for every render below
    R.render(big.cameras, 8, wl.depth, 0, xyz=False)
    out = {"out_spectral": torch.empty((wl.n_pixels, 16), dtype=torch.float64, device="cuda"),
           "out_xyz": torch.empty((wl.n_pixels, 3), dtype=torch.float32, device="cuda")}

    def captured():
        for o in out.values():
            o.fill_(-1.0)
        R.render(wl.cameras, 1, wl.depth, 3, use_graph=True, **opts, **out)
        return [o.clone() for o in out.values()]

    first = captured()
    assert all(torch.equal(a, b) for a, b in zip(captured(), first))
    # the four-band state, or the guide's queues, are allocated anew
    if between == "more_samples":
        R.render(wl.cameras, 16, wl.depth, 4, xyz=False, **opts)
    else:
        R.render(big.cameras, 2, wl.depth, 4, xyz=False, **opts)
    assert all(torch.equal(a, b) for a, b in zip(captured(), first))
