"""Rays whose directions are not of unit length, up to the largest floats: the
hit triangle is that of the unit direction."""
import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-20, 0, 100, 126, 127])
@pytest.mark.parametrize("builder", [1, 2])
def test_direction_length(exponent, builder):
    from paper_1912_04000_gb300.renderer import Renderer

    wl = scenes.prism_room()
    R = Renderer(0).load(wl, builder=builder)
    rng = np.random.default_rng(5)
    o, d = scenes.random_rays(rng, wl.scene, 20000)
    _, p1 = (a.cpu().numpy() for a in R.trace_closest(o, d))
    # (a power of two scales every component without rounding)
    t, p = (a.cpu().numpy() for a in R.trace_closest(o, np.ldexp(d, exponent)))
    assert (p1 >= 0).all()
    # (distances below the normal range are coarse: two hits near each other
    # may change places)
    assert (p == p1).mean() > 0.9995 and (p >= 0).all() and (t > 0.0).all()
    sun = np.zeros(len(d), int)
    _, g1 = (a.cpu().numpy() for a in R.trace_shadow(o, d, sun))
    _, g = (a.cpu().numpy() for a in R.trace_shadow(o, np.ldexp(d, exponent), sun))
    assert (g == g1).mean() > 0.9995
