"""The default NLOS kernels (samples in the order of the hidden surface, warps of neighbouring sensors) against the
general kernel, which a launch configuration with aggregation or privatised bins selects: the same connections, so
the same films up to the order of additions."""
import numpy as np
import pytest

from gpu_util import build_and_load, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5  # sums of up to 4200 FP32 terms of one sign in another order: sqrt(4200) * 6e-8 per bin


@pytest.fixture(scope="module")
def nlos(scenes_mod):
    api = build_and_load()
    return api, api.Scene(scenes_mod.nlos_scene())


def _both(api, s, kind, L, S, mode, T, spp, seed, flags=0, off=0):
    import torch
    rows = L.shape[0] * (S.shape[0] if S is not None else 1)
    res = []
    for opt in (0, api.MT_OPT_AGGREGATE):
        s.set_launch(kind, 256, 32 if kind == api.MT_LAUNCH_NLOS_EXHAUSTIVE else 1, 0, 0, opt)
        out = (torch.full((rows, T), 0.5, device="cuda"), torch.full((rows,), 0.25, device="cuda"))
        api.render_nlos(s, L, S, mode, T, 0.0, 12.288 / T, spp, seed, sample_offset=off, flags=flags, out=out)
        s.sync()
        res.append([x.cpu().numpy().astype(np.float64) for x in out])
    s.set_launch(kind, 256, 32 if kind == api.MT_LAUNCH_NLOS_EXHAUSTIVE else 1, 0, 0, 0)
    (f, st), (rf, rs) = res
    assert np.abs(rf).max() > 0 or rows * spp < 100  # a single sample may be occluded
    assert rel_l2(f, rf) < TOL and rel_l2(st, rs) < TOL


# samples per point around the batch of 1024 and below the ordering's least; rows that make the total large enough
@pytest.mark.parametrize("rows,spp", [(2048, 256), (520, 1023), (512, 1024), (512, 1025), (130, 4100), (37, 255), (3, 1)])
def test_scan_points(nlos, scenes_mod, rows, spp):
    import torch
    api, s = nlos
    L = torch.from_numpy(scenes_mod.wall_grid(rows, 1)).cuda()
    _both(api, s, api.MT_LAUNCH_NLOS, L, None, api.MT_CONFOCAL, 300, spp, 7)


# sensors around a warp and the ordering's cells, runs of 4 to 128 samples, with and without the ordering
@pytest.mark.parametrize("nl,ns,spp", [(1, 1, 1), (2, 31, 70), (3, 33, 255), (5, 64, 1024), (2, 2500, 1025), (300, 65, 300),
                                       (1, 4096, 1030)])
def test_pairs(nlos, scenes_mod, nl, ns, spp):
    import torch
    api, s = nlos
    L = torch.from_numpy(scenes_mod.wall_grid(nl, 1)).cuda()
    w = int(np.ceil(np.sqrt(ns)))
    S = torch.from_numpy(scenes_mod.wall_grid(w, w)[:ns].copy()).cuda()
    _both(api, s, api.MT_LAUNCH_NLOS_EXHAUSTIVE, L, S, api.MT_EXHAUSTIVE, 200, spp, 9)


@pytest.mark.parametrize("mode", ["scan", "pairs"])
def test_accumulation_and_offset(nlos, scenes_mod, mode):
    import torch
    api, s = nlos
    L = torch.from_numpy(scenes_mod.wall_grid(32, 32)).cuda()
    if mode == "scan":
        _both(api, s, api.MT_LAUNCH_NLOS, L, None, api.MT_CONFOCAL, 128, 512, 5, flags=api.MT_ACCUMULATE, off=1000)
    else:
        _both(api, s, api.MT_LAUNCH_NLOS_EXHAUSTIVE, L[:9].contiguous(), L, api.MT_EXHAUSTIVE, 128, 512, 5,
              flags=api.MT_ACCUMULATE, off=1000)


def test_sensors_at_one_point_and_on_a_line(nlos, scenes_mod):
    """The sensor order's extent is empty in one or both axes."""
    import torch
    api, s = nlos
    L = torch.from_numpy(scenes_mod.wall_grid(4, 4)).cuda()
    one = torch.zeros((500, 3), device="cuda")
    line = torch.from_numpy(scenes_mod.wall_grid(500, 1)).cuda()
    for S in (one, line):
        _both(api, s, api.MT_LAUNCH_NLOS_EXHAUSTIVE, L, S, api.MT_EXHAUSTIVE, 128, 600, 5)
