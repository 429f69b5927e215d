"""Exhaustive captures with few sensors or samples, on both sides of the lines between the kernel that gives a warp 32 sensors and
the one that gives every lane a pair: the same film as an aggregating launch, which takes neither rule."""
import numpy as np
import pytest

from gpu_util import build_and_load

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nlos(scenes_mod):
    api = build_and_load()
    return api, api.Scene(scenes_mod.nlos_scene())


# at most 16 sensors and 32 lasers per sensor; 64 beyond 4096 samples; any number up to 32 samples; at most 12 samples
# and fewer than 2^18 connections; one sensor and at most 1024
@pytest.mark.parametrize("nl,ns,spp", [(1, 16, 32), (1, 17, 32), (3, 5, 33), (1, 1, 1024), (1, 1, 1025), (31, 1, 1025), (32, 1, 1100), (64, 2, 4096),
                                       (63, 1, 4097), (64, 1, 4097), (511, 16, 64), (512, 16, 64), (544, 17, 64),
                                       (1, 40, 12), (1, 40, 13), (575, 40, 11), (576, 40, 12)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_few_sensors(nlos, scenes_mod, nl, ns, spp, accumulate):
    import torch
    api, s = nlos
    L = torch.from_numpy(scenes_mod.wall_grid(24, 24)[:nl].copy()).cuda()
    S = torch.from_numpy(scenes_mod.wall_grid(7, 7)[:ns].copy()).cuda()
    T, res = 200, []
    for opt in (0, api.MT_OPT_AGGREGATE):
        s.set_launch(api.MT_LAUNCH_NLOS_EXHAUSTIVE, 256, 32, 0, 0, opt)
        out = (torch.full((nl * ns, T), 0.5, device="cuda"), torch.full((nl * ns,), 0.25, device="cuda"))
        api.render_nlos(s, L, S, api.MT_EXHAUSTIVE, T, 0.0, 12.288 / T, spp, 3, out=out,
                        flags=api.MT_ACCUMULATE if accumulate else 0)
        s.sync()
        res.append([x.cpu().numpy().astype(np.float64) for x in out])
    for got, want in zip(*res):  # sums of at most 4097 terms of one sign: 4098 * 2^-24 at worst
        assert want.max() > 0 and np.all(np.abs(got - want) <= 2.5e-4 * want)
