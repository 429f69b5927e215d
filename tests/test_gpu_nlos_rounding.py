"""Every NLOS kernel computes a connection with the same rounding: the default kernels (samples in the order of the
hidden surface, warps of neighbouring sensors) against the general kernel, which an aggregating launch configuration
selects, and against the contribution records of the dump."""
import numpy as np
import pytest

from gpu_util import build_and_load

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nlos(scenes_mod):
    api = build_and_load()
    return api, api.Scene(scenes_mod.nlos_scene())


def _render(api, s, L, S, T, start, width, spp, seed, opt, out):
    exh = S is not None
    s.set_launch(api.MT_LAUNCH_NLOS_EXHAUSTIVE if exh else api.MT_LAUNCH_NLOS, 256, 32 if exh else 1, 0, 0, opt)
    api.render_nlos(s, L, S, api.MT_EXHAUSTIVE if exh else api.MT_CONFOCAL, T, start, width, spp, seed, out=out)
    s.sync()
    return out


# 268 M connections in bins narrow enough that most bins hold one: a path length whose last bit differs moves its
# connection to the next bin.  One moved connection of 67 M in the film is about 1.2e-4 of the film's norm or more.
# A film bin adds few terms of one sign (1e-6 is 16 roundings), a steady value at most 1024 (sqrt(1024) * 2^-24 = 2e-6,
# twice over).
@pytest.mark.parametrize("seed", [1, 8])
def test_exhaustive_capture_of_full_size(nlos, scenes_mod, seed):
    import torch
    api, s = nlos
    L = torch.from_numpy(scenes_mod.wall_grid(16, 16)).cuda()
    S = torch.from_numpy(scenes_mod.wall_grid(32, 32)).cuda()
    T, rows = 4096, 256 * 1024
    got, want = [_render(api, s, L, S, T, 0.0, 12.288 / T, 1024, seed, opt,
                         (torch.empty((rows, T), device="cuda"), torch.empty(rows, device="cuda")))
                 for opt in (0, api.MT_OPT_AGGREGATE)]
    d2 = n2 = 0.0
    for i in range(0, rows, 16384):
        f, r = got[0][i:i + 16384], want[0][i:i + 16384]
        d2 += float((f - r).double().square().sum())
        n2 += float(r.double().square().sum())
    assert n2 > 0 and (d2 / n2) ** 0.5 < 1e-6
    assert float((got[1] - want[1]).double().norm() / want[1].double().norm()) < 4e-6


# Bins of one unit in the last place of a path length in [2, 4): the nonzero bins are the path lengths themselves.
# Samples per laser around the batch of 1024 and below the ordering's least; confocal above and below its own; the wall
# as it is and tilted, with points off every axis.
@pytest.mark.parametrize("tilted", [False, True])
@pytest.mark.parametrize("nl,ns,spp", [(3, 7, 255), (3, 7, 256), (2, 11, 1025), (1, 33, 1024), (9, 0, 100), (64, 0, 8192)])
def test_path_lengths_to_the_last_bit(scenes_mod, nl, ns, spp, tilted):
    import torch
    api = build_and_load()
    sc = scenes_mod.nlos_scene()
    rng = np.random.default_rng(nl + ns)
    move = np.float32(0.05 if tilted else 0.0)
    if tilted:
        w = np.array([0.1, 0.25, np.sign(sc.wall["normal"][2])])
        sc.wall = dict(sc.wall, normal=tuple(float(x) for x in w / np.linalg.norm(w)))

    def points(g, n):
        p = scenes_mod.wall_grid(g, g)
        p = p[np.linspace(0, len(p) - 1, n).astype(int)]
        return torch.from_numpy((p + move * rng.uniform(-1, 1, p.shape)).astype(np.float32)).cuda()

    s = api.Scene(sc)
    L, S = points(8, nl), points(32, ns) if ns else None
    T, width = 1 << 23, 2.0 ** -22
    rows = nl * max(ns, 1)
    found = []
    for opt in (0, api.MT_OPT_AGGREGATE):
        film = _render(api, s, L, S, T, 2.0, width, spp, 5, opt,
                       (torch.empty((rows, T), device="cuda"), torch.empty(rows, device="cuda")))[0]
        at = film.nonzero()
        found.append((at.cpu().numpy(), film[at[:, 0], at[:, 1]].cpu().numpy().astype(np.float64)))
        del film
    (at, v), (r_at, r_v) = found
    assert len(r_at) > 0 or nl == 1  # a single laser point may see no hidden sample
    assert np.array_equal(at, r_at)
    assert np.all(np.abs(v - r_v) <= 2.0 ** -22 * r_v)  # a bin that several connections share adds them in any order
    if rows * spp <= 1 << 16:
        mode = api.MT_EXHAUSTIVE if ns else api.MT_CONFOCAL
        rec = api.render_dump(s, 1, 1, 64, 2.0, 1.0, spp, 5, 2, rows * spp, scan_args=(L, S, mode))[2]
        rec = rec[(rec["opl"] >= 2.0) & (rec["opl"] < 4.0)]
        bins = ((rec["opl"].astype(np.float64) - 2.0) / width).astype(np.int64)
        assert np.array_equal(np.unique(rec["pixel"].astype(np.int64) * T + bins), np.unique(r_at[:, 0] * T + r_at[:, 1]))
