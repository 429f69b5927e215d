"""The default exhaustive capture takes the sensors in an order it computes: every sensor once, wherever they lie.
Against the general kernel (which an aggregating launch configuration selects) that takes them as given."""
import numpy as np
import pytest

from gpu_util import build_and_load

pytestmark = pytest.mark.gpu

SPP = 4096  # with 1024 or more pairs: the smallest number of connections from which the sensors are put in order


def _sensors(kind, n):
    if kind == "cell edges":  # a grid of n points per side whose every coordinate is a border of the 32 cells
        u = np.linspace(-1.0, 1.0, n, dtype=np.float32)
        p = np.stack(np.meshgrid(u, u), -1).reshape(-1, 2)
    elif kind == "near edges":  # the neighbours of those borders in float
        k = np.arange(n) % 33
        e = np.float32(-1.0) + np.float32(2.0) * k.astype(np.float32) / np.float32(32.0)
        side = np.where(np.arange(n) % 3 == 0, np.float32(-2), np.float32(2))
        p = np.stack([np.nextafter(e, side), np.nextafter(e[::-1], side[::-1])], -1).astype(np.float32)
    else:  # scattered, with two points that no cell holds
        p = np.random.default_rng(n).uniform(-1.0, 1.0, (n, 2)).astype(np.float32)
        p[n // 3] = np.nan
        p[n // 2] = np.inf
    return np.concatenate([p, np.zeros((len(p), 1), np.float32)], 1)


# tilted: the two axes across the wall normal are no coordinate axes, so the cell is a rounded sum of products
@pytest.mark.parametrize("tilted", [False, True])
@pytest.mark.parametrize("kind,n", [("cell edges", 17), ("cell edges", 33), ("near edges", 1000), ("scattered", 65),
                                    ("scattered", 3001)])
def test_every_sensor_once(scenes_mod, kind, n, tilted):
    import torch
    api = build_and_load()
    sc = scenes_mod.nlos_scene()
    if tilted:
        w = np.array([0.1, 0.25, np.sign(sc.wall["normal"][2])])
        sc.wall = dict(sc.wall, normal=tuple(float(x) for x in w / np.linalg.norm(w)))
    s = api.Scene(sc)
    L = torch.from_numpy(scenes_mod.wall_grid(4, 4)).cuda()
    S = torch.from_numpy(_sensors(kind, n)).cuda()
    rows = 16 * S.shape[0]
    res = []
    for opt in (0, api.MT_OPT_AGGREGATE):
        s.set_launch(api.MT_LAUNCH_NLOS_EXHAUSTIVE, 256, 32, 0, 0, opt)
        film, steady = api.render_nlos(s, L, S, api.MT_EXHAUSTIVE, 1, 0.0, 100.0, SPP, 3)
        s.sync()
        res.append((film.cpu().numpy()[:, 0].astype(np.float64), steady.cpu().numpy().astype(np.float64)))
    (f, st), (rf, rs) = res
    assert (rs > 0).sum() > rows // 2
    # a row is a sum of at most 4096 terms of one sign, in another order: 4096 * 2^-24 at worst
    for got, want in ((f, rf), (st, rs)):
        assert np.all(np.abs(got - want) <= 2.5e-4 * want)
