"""Frequency-space and Stokes films that start 0 to 3 floats past a 16-byte boundary: the wavefront form adds pairs and
quads of floats only where the film allows it; the sums are the same up to their order."""
import numpy as np
import pytest

from gpu_util import build_and_load, rel_l2

pytestmark = pytest.mark.gpu


def _at(n, off):
    import torch
    return torch.empty(n + 8, dtype=torch.float32, device="cuda")[off:off + n]


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("kind", ["phasor1", "phasor3", "phasor4", "stokes"])
def test_film_offsets(scenes_mod, kind, off):
    import torch
    api = build_and_load()
    s = api.Scene(scenes_mod.diff_scene())  # conductors: every Stokes component
    s.set_launch(api.MT_LAUNCH_RENDER, 256, 1, 0, 0, api.MT_OPT_WAVEFRONT)
    H, W, spp, seed, depth = 17, 23, 8, 5, 6
    res = []
    for o in (0, off):
        if kind == "stokes":
            film = _at(H * W * 64 * 12, o).view(H, W, 64, 4, 3)
            steady = _at(H * W * 12, o).view(H, W, 4, 3)
            api.render_polarized(s, H, W, 64, 12.0, 0.1, spp, seed, depth, out=(film, steady))
        else:
            K = int(kind[-1])
            lam = torch.tensor([0.4 / 2 ** k for k in range(K)], device="cuda")
            film = _at(H * W * 2 * K * 3, o).view(H, W, 2 * K, 3)
            steady = _at(H * W * 3, o).view(H, W, 3)
            f = api.Film(film, steady, 0.0, 1.0)
            api.mt_render_phasor(s.h, f.h, api._ptr(lam), K, spp, seed, depth, 0, api._stream())
        s.sync()
        res.append((film.cpu().numpy().astype(np.float64), steady.cpu().numpy().astype(np.float64)))
    (a, sa), (b, sb) = res
    assert np.abs(a).max() > 0
    # at most 8 x 11 FP32 terms per entry in another order: 88 roundings of 6e-8 of the largest partial sum
    assert rel_l2(b, a) < 1e-5 and rel_l2(sb, sa) < 1e-5
