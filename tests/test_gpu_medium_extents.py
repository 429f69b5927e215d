"""Media in boxes of extreme extents: half-open and huge boxes around the room are the homogeneous medium that a box of
ordinary size around it is, and a box too thin to hold a point scatters nothing."""
import numpy as np
import pytest

from gpu_util import build_and_load, rel_l2

pytestmark = pytest.mark.gpu


def _render(api, scenes_mod, lo, hi, form):
    sc = scenes_mod.cornell_box()
    if lo is not None:
        # the density of a homogeneous grid is its value wherever the lookup lands
        sc.medium = dict(lo=lo, hi=hi, density=np.full((3, 4, 5), 0.5, np.float32), albedo=0.9, g=0.3)
    s = api.Scene(sc)
    if form == "wavefront":
        s.set_launch(api.MT_LAUNCH_RENDER, 256, 1, 0, 0, api.MT_OPT_WAVEFRONT)
    film, steady = api.render(s, 32, 32, 64, 3.0, 0.1, 16, 5, 6)
    s.sync()
    return film.cpu().numpy(), steady.cpu().numpy()


@pytest.mark.parametrize("form", ["megakernel", "wavefront"])
@pytest.mark.parametrize("lo,hi", [(-50.0, float("inf")), (-2e38, 2e38), (-1e38, 1e38), (-1e30, 1e30)])
def test_huge_boxes(scenes_mod, lo, hi, form):
    api = build_and_load()
    film, steady = _render(api, scenes_mod, (lo,) * 3, (hi,) * 3, form)
    ref, ref_s = _render(api, scenes_mod, (-50.0,) * 3, (50.0,) * 3, form)
    # the same paths; a weighted mean of equal densities is the density up to three roundings, over tens of lookups
    assert np.isfinite(film).all() and ref_s.max() > 0
    assert rel_l2(steady, ref_s) < 1e-4 and rel_l2(film, ref) < 1e-4


@pytest.mark.parametrize("form", ["megakernel", "wavefront"])
def test_a_box_thinner_than_any_step(scenes_mod, form):
    api = build_and_load()
    film, steady = _render(api, scenes_mod, (0.0, 0.0, 0.0), (1e-39, 1e-39, 1e-39), form)
    assert np.isfinite(film).all() and np.isfinite(steady).all() and steady.max() > 0
