"""render() through the native autograd node against the Python autograd
function it stands in for: the same bits, the same refusals."""
import math

import numpy as np
import pytest

from paper_2508_06768_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _case(dtype, **kw):
    import torch
    vol = I.small_phantom(n=40, seed=9)
    fan = I.Fan(33, 150, math.radians(55), 33.0, 5.0, 0.5)
    v = torch.from_numpy(vol.data).cuda().to(dtype)
    p = torch.from_numpy(I.top_face_pose(vol)).cuda()
    return v, p, fan, I.Params(seed=3, mode=1, **kw)


def _grads(fn, v, p, wrt_v, wrt_p):
    import torch
    v = v.clone().requires_grad_(wrt_v)
    p = p.clone().requires_grad_(wrt_p)
    img, valid = fn(v, p)
    assert not valid.requires_grad
    G = torch.from_numpy(I.random_weights(tuple(img.shape), 1)).cuda()
    wrt = [t for t, w in ((v, wrt_v), (p, wrt_p)) if w]
    return img.detach(), valid, torch.autograd.grad(img, wrt, G)


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
@pytest.mark.parametrize("wrt", [(True, True), (True, False), (False, True)])
@pytest.mark.parametrize("kw", [{}, {"atten": 1}, {"blur": 0, "speckle": 0}, {"refine": 1}])
def test_native_node_equals_python_function(dtype, wrt, kw):
    import torch
    from paper_2508_06768_gb300 import render as R
    v, p, fan, prm = _case(getattr(torch, dtype), **kw)
    sp, org = (1.0, 1.1, 0.9), (0.5, -0.25, 0.0)
    assert R._native_call(v, p, fan, prm, sp, org, 7) is not None
    a = _grads(lambda x, y: R.render(x, y, fan, prm, spacing=sp, origin=org, pose_ctr=7), v, p, *wrt)
    b = _grads(lambda x, y: R._Render.apply(x, y, sp, org, fan, prm, 7), v, p, *wrt)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    for x, y in zip(a[2], b[2]):
        assert x.dtype == y.dtype and torch.equal(x, y)


def test_native_node_strides_graph_and_refusals():
    import torch
    from paper_2508_06768_gb300 import binding as B
    from paper_2508_06768_gb300 import render as R
    v, p, fan, prm = _case(torch.float32)
    # a permuted volume and a double pose are copied, as before
    img, _ = R.render(v.permute(2, 1, 0), p.double(), fan, prm)
    ref, _, _ = B.render_fwd(v.permute(2, 1, 0).contiguous(), (1.0,) * 3, (0.0,) * 3, p, fan, prm)
    assert torch.equal(img, ref)
    # an expanded output gradient
    q = p.clone().requires_grad_()
    R.render(v, q, fan, prm)[0].sum().backward()
    q2 = p.clone().requires_grad_()
    R._Render.apply(v, q2, (1.0,) * 3, (0.0,) * 3, fan, prm, 0)[0].sum().backward()
    assert torch.equal(q.grad, q2.grad)
    # saved tensors: hooks see them, in-place changes are caught, a second backward is refused
    seen = []
    q = p.clone().requires_grad_()
    with torch.autograd.graph.saved_tensors_hooks(lambda t: seen.append(tuple(t.shape)) or t, lambda t: t):
        out = R.render(v, q, fan, prm)[0]
    assert sorted(seen) == sorted([tuple(v.shape), (6,)])
    out.sum().backward()
    with pytest.raises(RuntimeError):
        out.sum().backward()
    w = v.clone().requires_grad_()
    out = R.render(w, q, fan, prm)[0]
    with torch.no_grad():
        w.mul_(1.0)
    with pytest.raises(RuntimeError, match="modified by an inplace"):
        out.sum().backward()
    # errors of the C ABI keep their type; transforms and other devices are refused as before
    with pytest.raises(B.DiffusError):
        R.render(v, p, I.Fan(0, 5, 1.0, 10.0), prm)
    with pytest.raises(B.DiffusError):
        R.render(v, p, fan, prm.with_(mode=3))
    with pytest.raises(B.DiffusError):
        R.render(v.half(), p, fan, prm)
    with pytest.raises(B.DiffusError):
        R.render(v.cpu(), p.cpu(), fan, prm)
    with pytest.raises(RuntimeError):
        torch.func.grad(lambda y: R.render(v, y, fan, prm)[0].sum())(p)
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda y: R.render(v, y, fan, prm)[0])(p[None].repeat(2, 1))
    with pytest.raises(Exception):
        with torch.autograd.forward_ad.dual_level():
            R.render(v, torch.autograd.forward_ad.make_dual(p, torch.ones_like(p)), fan, prm)


def test_native_node_on_side_streams_and_threads():
    import threading

    import torch
    from paper_2508_06768_gb300 import render as R
    v, p, fan, prm = _case(torch.float32)
    ref = _grads(lambda x, y: R.render(x, y, fan, prm), v, p, True, True)
    torch.cuda.synchronize()
    got = [None] * 4

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(10):
                got[i] = _grads(lambda x, y: R.render(x, y, fan, prm), v, p, True, True)
        s.synchronize()

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    for g in got:
        assert torch.equal(g[0], ref[0])
        assert all(torch.equal(x, y) for x, y in zip(g[2], ref[2]))
