"""render() under compiled autograd: the backward pass is traced, with whatever
the node keeps, and gives the gradients of the plain one."""
import math

import pytest

from paper_2508_06768_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_backward_under_compiled_autograd():
    import torch
    import torch._dynamo.compiled_autograd as ca
    from paper_2508_06768_gb300 import render as R
    vol = I.small_phantom(n=40, seed=9)
    # a seed and angles whose bytes are no text
    prm = I.Params(seed=2**63 + 0xF0C1, mode=1)
    v0 = torch.from_numpy(vol.data).cuda()
    p0 = torch.from_numpy(I.top_face_pose(vol)).cuda()

    def grads(fan, compiled):
        v, p = v0.clone().requires_grad_(), p0.clone().requires_grad_()
        img, valid = R.render(v, p, fan, prm)
        assert R._native_call(v, p, fan, prm, (1.0,) * 3, (0.0,) * 3, 0) is not None and not valid.requires_grad
        G = torch.from_numpy(I.random_weights(tuple(img.shape), 1)).cuda()
        if compiled:
            with ca._enable(lambda gm: torch.compile(gm, backend="eager")):
                img.backward(G)
        else:
            img.backward(G)
        return v.grad, p.grad

    # calls of the same shapes and of others, so that nothing kept is taken for a constant
    for fan in (I.Fan(33, 150, math.radians(55), 33.0, 5.0, 0.5), I.Fan(33, 150, math.radians(35), 30.0, 5.0, 0.5),
                I.Fan(20, 99, math.radians(55), 33.0, 5.0, 0.5)):
        for a, b in zip(grads(fan, False), grads(fan, True)):
            assert torch.equal(a, b)


def test_image_without_a_gradient():
    # a function downstream that passes no gradient on: zeros, as from the Python function
    import torch
    from paper_2508_06768_gb300 import render as R

    class Stop(torch.autograd.Function):
        @staticmethod
        def forward(ctx, x):
            return x.sum()

        @staticmethod
        def backward(ctx, g):
            return None

    vol, prm = I.small_phantom(n=40, seed=9), I.Params(seed=3, mode=1)
    fan = I.Fan(33, 150, math.radians(55), 33.0, 5.0, 0.5)
    for f in (lambda v, p: R.render(v, p, fan, prm),
              lambda v, p: R._Render.apply(v, p, (1.0,) * 3, (0.0,) * 3, fan, prm, 0)):
        v = torch.from_numpy(vol.data).cuda().requires_grad_()
        p = torch.from_numpy(I.top_face_pose(vol)).cuda().requires_grad_()
        gv, gp = torch.autograd.grad(Stop.apply(f(v, p)[0]), (v, p))
        assert not gv.any() and not gp.any() and gv.shape == v.shape and gp.shape == (6,)
