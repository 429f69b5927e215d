"""TransientRender's backward pass where one output's gradient, or neither, is defined, and whose memory its gradients
are."""
import numpy as np
import pytest

from gpu_util import build_and_load

pytestmark = pytest.mark.gpu

ARGS = (16, 20, 64, 3.5, 0.04, 4, 7, 4)


@pytest.fixture(scope="module")
def setup(scenes_mod):
    import torch
    api = build_and_load()
    sc = scenes_mod.cornell_box()
    return (api, api.Scene(sc), torch.from_numpy(sc.albedo).cuda().requires_grad_(True),
            torch.tensor([list(e["radiance"]) for e in sc.emitters], device="cuda", requires_grad=True))


def test_undefined_output_gradients_give_zeros(setup):
    import torch
    api, s, alb, rad = setup

    class Undefined(torch.autograd.Function):
        @staticmethod
        def forward(ctx, x):
            return x.sum()

        @staticmethod
        def backward(ctx, g):
            return None
    film, steady = api.TransientRender.apply(alb, rad, s, *ARGS)
    grads = torch.autograd.grad(Undefined.apply(film) + Undefined.apply(steady), (alb, rad))
    assert [tuple(g.shape) for g in grads] == [tuple(alb.shape), tuple(rad.shape)]
    assert all(float(g.abs().max()) == 0.0 for g in grads)


@pytest.mark.parametrize("used", ["film", "steady"])
def test_one_output_used(setup, used):
    import torch
    api, s, alb, rad = setup
    film, steady = api.TransientRender.apply(alb, rad, s, *ARGS)
    only = torch.autograd.grad((film if used == "film" else steady).sum(), (alb, rad))
    film, steady = api.TransientRender.apply(alb, rad, s, *ARGS)
    both = torch.autograd.grad(film.sum() * (used == "film") + steady.sum() * (used == "steady"), (alb, rad))
    for a, b in zip(only, both):
        assert float(b.abs().max()) > 0 and np.allclose(a.cpu(), b.cpu(), rtol=1e-4, atol=1e-6 * float(b.abs().max()))


def test_gradients_own_their_memory(setup):
    import torch
    api, s, alb, rad = setup
    g = api.render_backward(s, 64, 3.5, 0.04, 4, 7, 4, torch.ones((16, 20, 64, 3), device="cuda"))
    for t in g:
        assert t._base is None and t.untyped_storage().nbytes() == 4 * t.numel()
    assert len({t.untyped_storage().data_ptr() for t in g}) == 3
