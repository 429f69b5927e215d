"""A launch configuration set without arguments is that of a new scene, and a film with every bin privatised is the
default's up to the order of additions."""
import numpy as np
import pytest

from gpu_util import build_and_load, rel_l2

pytestmark = pytest.mark.gpu

H, W, T, START, WIDTH, SPP, SEED, DEPTH = 64, 64, 256, 3.5, 0.01, 16, 25660, 4


def _render(api, s, flags=0):
    s.read_counters()
    film, steady = api.render(s, H, W, T, START, WIDTH, SPP, SEED, DEPTH, flags=flags)
    c = s.read_counters()
    return film.cpu().numpy(), steady.cpu().numpy(), c


def test_render(scenes_mod):
    api = build_and_load()
    s = api.Scene(scenes_mod.cornell_box())
    new = _render(api, s, api.MT_COUNTERS)[2]
    s.set_launch(api.MT_LAUNCH_RENDER, 256, 1, 0, -1, api.MT_OPT_AGGREGATE)
    s.set_launch(api.MT_LAUNCH_RENDER)
    film, steady, reset = _render(api, s, api.MT_COUNTERS)
    assert new["gmem_splats"] > 20000 and new["smem_splats"] == 0
    assert (reset["gmem_splats"], reset["smem_splats"]) == (new["gmem_splats"], 0)
    s.set_launch(api.MT_LAUNCH_RENDER, 256, 1, 0, T)  # D = T: 12 KB per one-pixel tile
    pf, ps, priv = _render(api, s, api.MT_COUNTERS)
    assert priv["gmem_splats"] == 0 and priv["smem_splats"] == new["gmem_splats"]
    plain = _render(api, s)
    for f, st in ((pf, ps), plain[:2]):  # a few hundred terms of one sign per entry at most
        assert rel_l2(f, film) < 1e-5 and rel_l2(st, steady) < 1e-5


@pytest.mark.parametrize("mode", ["confocal", "exhaustive"])
def test_nlos(scenes_mod, mode):
    import torch
    api = build_and_load()
    s = api.Scene(scenes_mod.nlos_scene())
    exh = mode == "exhaustive"
    L = torch.from_numpy(scenes_mod.wall_grid(8, 8)).cuda()
    S = torch.from_numpy(scenes_mod.wall_grid(16, 16)).cuda() if exh else None
    kind = api.MT_LAUNCH_NLOS_EXHAUSTIVE if exh else api.MT_LAUNCH_NLOS

    def run():
        n0 = s.stats()["launches"]
        film, steady = api.render_nlos(s, L, S, api.MT_EXHAUSTIVE if exh else api.MT_CONFOCAL, 4096, 0.0, 0.003, 300, 3)
        s.sync()
        return film.cpu().numpy(), steady.cpu().numpy(), s.stats()["launches"] - n0
    new = run()
    s.set_launch(kind, 128, 2, 1, -1, api.MT_OPT_AGGREGATE)
    priv = run()
    s.set_launch(kind)
    reset = run()
    # the default of an exhaustive grid of this size puts the sensors in order first: one more kernel than the general form
    assert new[2] == reset[2] == (3 if exh else 1) and priv[2] == (2 if exh else 1)
    for f, st, _ in (priv, reset):
        assert rel_l2(f, new[0]) < 1e-5 and rel_l2(st, new[1]) < 1e-5
