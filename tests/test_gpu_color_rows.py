"""The staged colour rows of the projection and its adjoint, for every row length
(3, 12, 27 and 48 floats) at partial warps, whose last floats are no whole float4."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_14244_gb300 import igs
from paper_2403_14244_gb300.render import Renderer

from . import _gpu
from ._tiny import random_small

pytestmark = pytest.mark.gpu

SIZES = [1, 3, 31, 32, 33, 61, 97]


def _setup(n, sh):
    sc, cam = random_small(n, 70 + n, w=48, h=40, sh_degree=sh, log_params=True)
    C = 3 if sh < 0 else 3 * (sh + 1) ** 2
    scene = igs.Scene(*(torch.from_numpy(np.ascontiguousarray(a)).cuda()
                        for a in (sc.means_sigma, sc.opacity, sc.color.reshape(n, C))))
    r = Renderer(tile=16, sh_degree=sh, param_mode=1)
    return sc, igs.camera(cam), cam, scene, r


@pytest.mark.parametrize("sh", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("n", SIZES)
def test_rows_forward_and_gradients(n, sh):
    sc, c, cam, scene, r = _setup(n, sh)
    img, f = r.run_forward(scene, c)
    ref = oracle.render(sc, cam, mode=1, flag_margin=2e-5)
    _gpu.compare_images(img.cpu().numpy().astype(np.float64), ref["img"], ref["flag"], max_flag_frac=0.02)
    W = np.random.default_rng(n).normal(size=(3, 40, 48)).astype(np.float32)
    # a colour gradient buffer that starts four bytes past a 16-byte boundary is taken when its rows
    # are no multiple of 16 bytes
    C = scene.color.shape[1]
    shift = 1 if C % 4 else 0
    d_col = torch.full((n * C + shift + 4,), 7.0, device="cuda")[shift:shift + n * C].view(n, C)
    grads = (torch.empty_like(scene.means_sigma), torch.empty_like(scene.opacity), d_col)
    d_ms, d_op, d_col = (t.cpu().numpy() for t in r.run_backward(scene, c, f, torch.from_numpy(W).cuda(), grads))
    g = oracle.backward(sc, cam, W.astype(np.float64), mode=1)
    _gpu.grad_close(d_ms[:, :3], g["d_means"], "means")
    _gpu.grad_close(d_col, g["d_color"].reshape(n, C), "color")


@pytest.mark.parametrize("sh", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("n", SIZES)
def test_rows_adam_and_next_projection(n, sh):
    """The fused projection backward + Adam moves rows and moments as the separate
    gradient and igs.adam do, writes nothing past them, and its next-view
    projection is that of the updated rows, bit for bit."""
    sc, c, cam, scene, r = _setup(n, sh)
    _, f = r.run_forward(scene, c)
    g2d = torch.randn((n, 8), device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(n)
    arrays = [scene.means_sigma, scene.opacity, scene.color]
    m0 = [0.1 * torch.randn(a.shape, generator=gen, device="cuda") for a in arrays]
    v0 = [0.01 + torch.rand(a.shape, generator=gen, device="cuda") for a in arrays]
    grads = [torch.empty_like(a) for a in arrays]
    igs.project_bwd(scene, c, r.opts, f, g2d, *grads)
    want = []
    for p, g, m, v in zip(arrays, grads, m0, v0):
        p, m, v = p.clone(), m.clone(), v.clone()
        igs.adam(p, g, m, v, 3, lr=1e-2)
        want.append((p, m, v))

    def padded(t):  # room behind the array, to see that nothing is written there
        buf = torch.full((t.numel() + 8,), 5.0, device="cuda")
        buf[:t.numel()] = t.reshape(-1)
        return buf, buf[:t.numel()].view(t.shape)
    bufs, views = zip(*(padded(t) for t in arrays + m0 + v0))
    fused = igs.Scene(*views[:3])
    state = torch.tensor([2, 0, 0, 0], dtype=torch.int32, device="cuda")
    nxt = igs.Frame(n, 1 << 14, c, r.opts)
    igs.project_bwd_adam_next(fused, c, r.opts, f, g2d, views[3:6], views[6:9], state, c, nxt, lr=1e-2)
    sep = igs.Frame(n, 1 << 14, c, r.opts)
    igs.project(fused, c, r.opts, sep)
    torch.cuda.synchronize()
    assert int(state[0]) == 3
    for k, (p, m, v) in enumerate(want):
        # both form the same FP32 update, one with approximate square root and division (a few 2^-22)
        torch.testing.assert_close(views[k], p, rtol=1e-5, atol=1e-6)
        torch.testing.assert_close(views[3 + k], m, rtol=1e-5, atol=1e-6)
        torch.testing.assert_close(views[6 + k], v, rtol=1e-5, atol=1e-6)
    for b in bufs:
        assert bool((b[-8:] == 5.0).all())
    for a, b in ((nxt.rec(), sep.rec()), (nxt.rect(), sep.rect()), (nxt.count(), sep.count()),
                 (nxt.depth_key(), sep.depth_key())):
        np.testing.assert_array_equal(a.cpu().numpy().view(np.uint32), b.cpu().numpy().view(np.uint32))
