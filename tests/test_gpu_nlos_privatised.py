"""Exhaustive captures with privatised bins and the automatic tile (as many sensors as have all their bins in 96 KB):
the same film as an aggregating launch, at the tile's edges."""
import numpy as np
import pytest

from gpu_util import build_and_load

pytestmark = pytest.mark.gpu


# tiles of 32, 32, 31, 6, 1 and 1 sensors (the last one's bins fit only in part)
@pytest.mark.parametrize("T", [100, 768, 770, 4096, 24576, 70000])
@pytest.mark.parametrize("priv", [-1, 50])
@pytest.mark.parametrize("accumulate", [False, True])
def test_automatic_tile(scenes_mod, T, priv, accumulate):
    import torch
    api = build_and_load()
    s = api.Scene(scenes_mod.nlos_scene())
    nl, ns, spp = 3, 40, 20
    L = torch.from_numpy(scenes_mod.wall_grid(3, 1)).cuda()
    S = torch.from_numpy(scenes_mod.wall_grid(8, 5)).cuda()
    res = []
    for p, opt in ((priv, 0), (0, api.MT_OPT_AGGREGATE)):
        s.set_launch(api.MT_LAUNCH_NLOS_EXHAUSTIVE, 0, 0, 0, p, opt)
        out = (torch.full((nl * ns, T), 0.5, device="cuda"), torch.full((nl * ns,), 0.25, device="cuda"))
        api.render_nlos(s, L, S, api.MT_EXHAUSTIVE, T, 0.0, 12.288 / T, spp, 3, out=out,
                        flags=api.MT_ACCUMULATE if accumulate else 0)
        s.sync()
        res.append([x.cpu().numpy().astype(np.float64) for x in out])
    for got, want in zip(*res):  # sums of at most 21 terms of one sign
        assert want.max() > 0 and np.all(np.abs(got - want) <= 21 * 2.0 ** -24 * want)
