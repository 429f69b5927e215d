"""GPU traversal at the edges of what the trees and the triangle records can hold, against closed forms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from gpu_util import build_and_load
    return build_and_load()


def _scene(api, tris):
    from paper_2510_25660_gb300 import scenes
    n = len(tris)
    return api.Scene(scenes.Scene(np.ascontiguousarray(tris, np.float32), np.full((n, 3), 0.5, np.float32),
                                  np.zeros(n, np.float32), np.zeros(n, np.uint32), [],
                                  dict(origin=(0, 0, 3), target=(0, 0, 0), up=(0, 1, 0), fov_x_deg=40.0)))


def _probe(api, s, o, d, **kw):
    import torch
    r = torch.from_numpy(np.concatenate([o, d], 1).astype(np.float32)).cuda()
    tri, t = api.probe_trace(s, r, **kw)
    return tri.cpu().numpy(), t.cpu().numpy()


@pytest.mark.parametrize("n", [5, 12, 24])
def test_deep_tree_fills_the_stack(api, n):
    """Triangles in the planes x = 8^-i: every split of the binned builder cuts off the outermost ones, so the tree
    is as deep as such a scene gets, and a ray along x through all of them pushes an entry at every level."""
    x = 8.0 ** -np.arange(n)
    tris = np.stack([np.stack([x, -np.ones(n), -np.ones(n)], 1), np.stack([x, np.ones(n), -np.ones(n)], 1),
                     np.stack([x, np.zeros(n), np.ones(n)], 1)], 1)
    s = _scene(api, tris)
    assert s.stats()["bvh_depth"] <= 62
    o = np.array([[2.0, 0, 0], [-x[-1], 0, 0], [2.0, 1e-3, 2e-3], [-x[-1], 1e-3, 2e-3], [2.0, 3.0, 0.0]])
    d = np.array([[-1.0, 0, 0], [1, 0, 0], [-1, 0, 0], [1, 0, 0], [-1, 0, 0]])
    want = [0, n - 1, 0, n - 1, -1]
    for wide in (False, True):
        tri, t = _probe(api, s, o, d, wide=wide)
        assert tri.tolist() == want
        assert np.allclose(t[:4], [1.0, 2 * x[-1], 1.0, 2 * x[-1]], rtol=1e-6, atol=0)
        occ, _ = _probe(api, s, o, d, any_hit=True, wide=wide)
        assert occ.tolist() == [1, 1, 1, 1, 0]


def test_every_axis_order_and_sign(api):
    """The six faces of a box, seen from inside along every dominant axis and sign: the row order of the
    triangle records and the test without the winding swap give the face and the distance of the closed form."""
    from paper_2510_25660_gb300 import scenes
    s = _scene(api, scenes.box_mesh((0.0, 0.0, 0.0), (2.0, 2.0, 2.0), 0.0))
    rng = np.random.default_rng(11)
    d = rng.normal(size=(4096, 3))
    d[:12] = np.concatenate([np.eye(3), -np.eye(3), np.eye(3)[[1, 2, 0]], -np.eye(3)[[1, 2, 0]]])
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32).astype(np.float64)
    o = rng.uniform(-0.5, 0.5, (4096, 3)).astype(np.float32).astype(np.float64)
    with np.errstate(divide="ignore"):
        tf = np.where(d > 0, (1 - o) / d, np.where(d < 0, (-1 - o) / d, np.inf))
    face = {(2, 1): 0, (2, -1): 1, (0, 1): 2, (0, -1): 3, (1, 1): 4, (1, -1): 5}
    ax = tf.argmin(1)
    want = np.array([face[(a, int(np.sign(d[i, a])))] for i, a in enumerate(ax)])
    srt = np.sort(tf, 1)
    clear = srt[:, 1] - srt[:, 0] > 1e-5  # away from the box's edges
    for wide in (False, True):
        tri, t = _probe(api, s, o, d, wide=wide)
        assert (tri[clear] // 2 == want[clear]).all()
        assert np.allclose(t[clear], tf.min(1)[clear], rtol=4e-6, atol=0)
        occ, _ = _probe(api, s, o, d, any_hit=True, tmax=0.49, wide=wide)
        assert not occ.any()
