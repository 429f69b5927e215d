"""Scenes of few triangles are traced triangle by triangle; counting renders (MT_COUNTERS) traverse the tree.  Same hits,
so the same films and gradients up to the order of additions, around the limits of the rule (8 to 48 triangles in a
medium, closed scenes of at most 48 without one) and for odd counts (triangles go in pairs)."""
import numpy as np
import pytest

from gpu_util import build_and_load, rel_l2

pytestmark = pytest.mark.gpu

# sums of at most a few thousand FP32 terms of one sign per entry in another order: sqrt(4000) * 6e-8
TOL = 1e-5


def _scene(scenes_mod, n, medium):
    """n triangles: a floor, a light above it, and random ones between."""
    rng = np.random.default_rng(n)
    floor = scenes_mod.quad((-2, -1, 2), (2, -1, 2), (2, -1, -2), (-2, -1, -2))
    light = np.array([[[-0.4, 1.4, -0.4], [0.4, 1.4, -0.4], [0.0, 1.4, 0.5]]])
    light = light if np.cross(light[0, 1] - light[0, 0], light[0, 2] - light[0, 0])[1] < 0 else light[:, ::-1]
    mesh = scenes_mod.random_mesh(n, max(n - 3, 0), 0.8)
    tris = np.concatenate([floor, light, mesh])[:n].astype(np.float32)
    alb = rng.uniform(0.2, 0.9, (n, 3)).astype(np.float32)
    em = [dict(type=0, first_tri=2, n_tris=1, radiance=(9.0, 8.0, 7.0))] if n >= 3 else \
         [dict(type=1, first_tri=0, n_tris=0, radiance=(5.0, 4.0, 3.0), position=(0.3, 1.0, 0.2))]
    sc = scenes_mod.Scene(tris, alb, np.zeros(n, np.float32), np.zeros(n, np.uint32), em,
                          dict(origin=(0, 0.2, 3.5), target=(0, -0.2, 0), up=(0, 1, 0), fov_x_deg=50.0))
    if medium:
        sc.medium = scenes_mod.homogeneous_medium(0.6, res=3)
    return sc


@pytest.mark.parametrize("form", ["megakernel", "wavefront"])
@pytest.mark.parametrize("case", ["1", "7m", "8m", "9m", "36", "47m", "48m", "49m", "cornell", "cornellm", "furnace"])
def test_triangle_loop_equals_tree(scenes_mod, case, form):
    import torch
    api = build_and_load()
    if case.startswith("cornell"):
        sc = scenes_mod.cornell_box()
        if case.endswith("m"):
            sc.medium = scenes_mod.homogeneous_medium(0.6, res=3)
    elif case == "furnace":
        sc = scenes_mod.furnace_sphere(0)
    else:
        sc = _scene(scenes_mod, int(case.rstrip("m")), case.endswith("m"))
    s = api.Scene(sc)
    opt = api.MT_OPT_WAVEFRONT if form == "wavefront" else 0
    for kind in (api.MT_LAUNCH_RENDER, api.MT_LAUNCH_BACKWARD):
        s.set_launch(kind, 256, 0, 0, 0, opt)
    H, W, T, start, width, spp, seed, depth = 40, 50, 64, 2.0, 0.2, 16, 5, 6
    film, steady = api.render(s, H, W, T, start, width, spp, seed, depth)
    ref, rsteady = api.render(s, H, W, T, start, width, spp, seed, depth, flags=api.MT_COUNTERS)
    g = torch.rand(film.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    grads = api.render_backward(s, T, start, width, spp, seed, depth, g)
    rgrads = api.render_backward(s, T, start, width, spp, seed, depth, g, flags=api.MT_COUNTERS)
    s.sync()
    assert float(rsteady.abs().max()) > 0
    for a, b in [(film, ref), (steady, rsteady)] + list(zip(grads, rgrads)):
        assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) < TOL
