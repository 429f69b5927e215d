"""Density lookups of participating media: odd grid shapes (cell records), and a grid too large for cell records
(read voxel by voxel), per contribution against the oracle."""
import numpy as np
import pytest

from gpu_util import build_and_load, match_contribs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["megakernel", "wavefront"])
@pytest.mark.parametrize("grid", ["3x5x7", "17x1x2", "fbm147"])
def test_density_grid_shapes(oracle_mod, scenes_mod, grid, form):
    api = build_and_load()
    if grid == "fbm147":  # 148^3 records would take 104 MB
        sc = scenes_mod.media_scene(res=147)
    else:
        res = tuple(int(x) for x in grid.split("x"))
        sc = scenes_mod.cornell_box()
        dens = np.random.default_rng(sum(res)).uniform(0.1, 2.0, res[::-1]).astype(np.float32)
        # extents that are no powers of two, a box that ends inside the room
        sc.medium = dict(lo=(-0.9, -0.7, -0.83), hi=(0.8, 0.95, 0.7), density=dens, albedo=0.9, g=0.3)
    s = api.Scene(sc)
    if form == "wavefront":
        s.set_launch(api.MT_LAUNCH_RENDER, 256, 0, 0, -1, api.MT_OPT_WAVEFRONT)
    H, W, T, start, width, spp, seed, depth = 24, 24, 256, 3.5, 0.02, 8, 17, 8
    _, _, rec, n = api.render_dump(s, H, W, T, start, width, spp, seed, depth, cap=1_000_000)
    s.sync()
    ref = oracle_mod.OracleScene(sc).render(H, W, T, start, width, spp, seed, depth, dump_cap=1_000_000)
    nm, div, worst, bad, bin_bad, _ = match_contribs(rec, ref["dump"], start=start, width=width)
    assert n == len(rec) and nm > 5000
    assert bin_bad == 0
    # the bounds of FP32 against FP64 on the 128^3 grid
    assert div <= 5e-4 * nm + 4 and bad <= 5e-3 * nm, (div, bad, nm, worst)


def test_division_by_a_known_divisor():
    """a * rc corrected once by its exact remainder is the correctly rounded a / c (the GPU's div_known): every
    product of two 24-bit significands and the remainder are exact in 64 bits."""
    rng = np.random.default_rng(5)
    c = rng.uniform(0.01, 100.0, 2_000_000).astype(np.float32)
    a = (rng.uniform(-1.0, 1.0, c.size) * 10.0 ** rng.uniform(-6, 3, c.size)).astype(np.float32)
    rc = np.float32(1.0) / c
    q = a * rc
    r = (a.astype(np.float64) - q.astype(np.float64) * c.astype(np.float64)).astype(np.float32)
    q1 = (q.astype(np.float64) + r.astype(np.float64) * rc.astype(np.float64)).astype(np.float32)
    assert (q1 == a / c).all()
