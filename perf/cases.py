"""What the framework is timed on: the work a user has it do, through its public entry points.

``listed()`` names twelve cases over the range of real use, from one frame of 4,096 Gaussians to a
32-view batch of two million; ``draw(rng)`` gives another case of the same ranges. ``prepare`` makes
a case's inputs on the GPU from a seed and whatever a program keeps between calls (renderer, training
state, batch, server); ``run`` is one pass; ``exact`` is the same result in 64-bit torch, written from
the definitions, where that is quick enough; ``work`` is what a pass cannot do without.

Sizes, distributions and cameras are those of ``scenes.py``, ``bench.py`` and the tests, drawn on the
GPU so that inputs are quick to make.
"""
import math

import numpy as np
import torch

from paper_2403_14244_gb300 import igs, scenes
from paper_2403_14244_gb300.batch import BatchRenderer
from paper_2403_14244_gb300.render import Renderer, TrainStep, render

DEV = "cuda"
EXACT_PAIRS = 1.2e10  # most (pixel, Gaussian) pairs that exact() evaluates densely (a few seconds)
FIT_LR = (2e-3, 2e-3, 2e-4, 2e-4, 2e-4, 2e-4, 0.0, 0.0)


def listed():
    return [
        # the smallest call: one frame of a small RGB scene, as an interactive viewer issues it (no status read)
        dict(name="render_4k_256", kind="render", n=4096, sh=-1, scene="uniform", width=256, height=256, tile=16,
             footprint=0, check=False),
        # an ordinary frame at odd sizes: SH degree 1, the call's defaults (frame status read back)
        dict(name="render_200k_odd", kind="render", n=200_003, sh=1, scene="clustered", width=1001, height=667,
             tile=16, footprint=0, check=True),
        # 1080p frame of a million Gaussians with degree-3 colours
        dict(name="render_1m_1080p", kind="render", n=1_000_000, sh=3, scene="clustered", width=1920, height=1080,
             tile=32, footprint=0, check=True),
        # a small differentiable render (pose or appearance fitting): forward and backward through autograd
        dict(name="grad_20k_320", kind="grad", n=20_011, sh=0, scene="clustered", width=320, height=240, tile=16),
        # forward and backward of the same million at 1080p
        dict(name="grad_1m_1080p", kind="grad", n=1_000_000, sh=3, scene="clustered", width=1920, height=1080, tile=32),
        # the training loop: one graph-replayed step (forward, L1, backward, Adam, next projection) at 3M Gaussians
        dict(name="train_3m", kind="train", n=3_000_000, sh=3, scene="uniform", width=1297, height=840, tile=32,
             ssim=0.0, graph=True),
        # the start of a training run: few Gaussians, eager steps, the loss with its structural term
        dict(name="train_30k_ssim", kind="train", n=30_000, sh=2, scene="uniform", width=401, height=299, tile=16,
             ssim=0.2, graph=False),
        # offline rendering of many views of mixed sizes in one captured chain
        dict(name="batch_2m_32", kind="batch", n=2_000_000, sh=3, scene="clustered", views=32, tile=32),
        # a burst of requests of mixed sizes to the render server, two resident scenes, four slots
        dict(name="serve_16", kind="serve", n=500_000, sh=3, scene="clustered", requests=16, tile=32),
        # the 2D experiment: one fitting iteration (render, loss, adjoint, Adam) of 1000 particles on 512 x 512
        dict(name="fit2d_1000", kind="fit2d", k=1000, width=512, height=512, D=15.0),
        # Gaussians from a coloured point set
        dict(name="octree_2m", kind="octree", n=2_000_000, levels=7, k_max=500_000, sh=-1),
        # the restructuring passes between training steps at full size: merge, and delete / divide
        dict(name="merge_3m", kind="merge", n=3_000_000, sh=3, cells=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "grad", "grad", "train", "train", "batch", "serve", "fit2d",
                       "octree", "merge", "densify"])
    sh = rng.choice([-1, 0, 1, 2, 3, 3])
    scene = rng.choice(["uniform", "clustered"])
    if kind == "octree":
        return dict(kind=kind, n=_log(rng, 20_000, 2_000_000), levels=rng.choice([5, 6, 7]),
                    k_max=_log(rng, 2_000, 500_000), sh=sh)
    if kind == "fit2d":
        return dict(kind=kind, k=_log(rng, 200, 4000), width=_log(rng, 96, 512), height=_log(rng, 96, 512),
                    D=rng.choice([15.0, 50.0]))
    if kind in ("merge", "densify"):
        return dict(kind=kind, n=_log(rng, 20_000, 3_000_000), sh=sh, cells=rng.choice([64, 128, 256]))
    if kind == "batch":
        return dict(kind=kind, n=_log(rng, 50_000, 1_000_000), sh=sh, scene=scene, views=rng.randint(3, 16),
                    tile=rng.choice([16, 32]))
    if kind == "serve":
        return dict(kind=kind, n=_log(rng, 50_000, 500_000), sh=sh, scene=scene, requests=rng.randint(4, 16),
                    tile=rng.choice([16, 32]))
    w = _log(rng, 200, 1920)
    c = dict(kind=kind, n=_log(rng, 1_000, 1_000_000), sh=sh, scene=scene, width=w,
             height=max(16, int(w * rng.uniform(0.5, 1.0))), tile=rng.choice([8, 16, 16, 32, 32]))
    if kind == "render":
        c.update(footprint=rng.choice([0, 0, 0, 1]), check=rng.choice([True, False]))
    if kind == "train":
        c.update(tile=rng.choice([16, 32]), ssim=rng.choice([0.0, 0.2]), graph=rng.choice([True, False]))
    return c


# ------------------------------------------------------------------ inputs --

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (int(seed) % (1 << 30)) + salt)
    return g


def _uniform(g, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV)


def _scene(case, seed, log_params=False):
    """means_sigma [n,4], opacity [n], color [n,C]: the uniform or clustered scene of scenes.py."""
    g, n, sh = _gen(seed), case["n"], case["sh"]
    if case.get("scene", "uniform") == "uniform":
        means = _uniform(g, (n, 3), -1.0, 1.0)
        sigma = torch.exp(_uniform(g, (n,), math.log(0.005), math.log(0.05)))
        op = _uniform(g, (n,), 0.05, 0.95)
    else:
        m = int(0.7 * n)
        centers, stds = _uniform(g, (64, 3), -1.0, 1.0), _uniform(g, (64,), 0.05, 0.3)
        which = torch.randint(0, 64, (m,), generator=g, device=DEV)
        shell = torch.nn.functional.normalize(torch.randn((n - m, 3), generator=g, device=DEV))
        means = torch.cat([centers[which] + torch.randn((m, 3), generator=g, device=DEV) * stds[which, None], shell])
        means = means[torch.randperm(n, generator=g, device=DEV)]
        sigma = torch.exp(math.log(0.01) + 0.7 * torch.randn((n,), generator=g, device=DEV))
        op = torch.sigmoid(1.5 * torch.randn((n,), generator=g, device=DEV))
    if sh < 0:
        col = torch.rand((n, 3), generator=g, device=DEV)
    else:
        col = 0.1 * torch.randn((n, 3 * (sh + 1) ** 2), generator=g, device=DEV)
        col[:, :3] = _uniform(g, (n, 3), -1.0, 1.0)
    if log_params:
        sigma, op = torch.log(sigma), torch.logit(op, eps=1e-6)
    return torch.cat([means, sigma[:, None]], 1).contiguous(), op.contiguous(), col.contiguous()


def _camera(seed, width, height, k=0):
    """A pinhole camera on a sphere of radius 4 looking at the origin."""
    r = np.random.default_rng([int(seed) % (1 << 30), k])
    a, e = r.uniform(0, 2 * math.pi), r.uniform(-0.4, 0.4)
    return scenes.pinhole((4 * math.cos(a) * math.cos(e), 4 * math.sin(e), 4 * math.sin(a) * math.cos(e)), width,
                          height, 0.85 * width)


def _image(seed, width, height, salt):
    return torch.rand((3, height, width), generator=_gen(seed, salt), device=DEV)


def _moments(seed, arrays, scale):
    """Adam moments as in the middle of a run: gradients of about `scale`."""
    g = _gen(seed, 77)
    m = [scale * 0.3 * torch.randn(a.shape, generator=g, device=DEV) for a in arrays]
    v = [(scale * (0.5 + torch.rand(a.shape, generator=g, device=DEV))) ** 2 for a in arrays]
    return m, v


def _train_scale(case):
    return 0.3 / (3 * case["width"] * case["height"])


TRAIN_T = 1000    # Adam steps taken before the measured one
TRAIN_LR = 1e-5   # late in a run: the scene, and so the work, stays the same from pass to pass
TRAIN_VIEWS = 4


def _serve_cameras(case, seed):
    res = scenes.RESOLUTIONS_SERVE
    return [_camera(seed, *res[k % len(res)], k=k) for k in range(case["requests"])]


def _batch_cameras(case, seed):
    res = scenes.RESOLUTIONS_BATCH
    return [_camera(seed, *res[k % len(res)], k=k) for k in range(case["views"])]


def _points(case, seed):
    """The coloured point set of scenes.point_cloud."""
    g, n = _gen(seed), case["n"]
    centres = _uniform(g, (64, 3), -0.8, 0.8)
    h = n // 2
    p = torch.cat([centres[torch.randint(0, 64, (h,), generator=g, device=DEV)] +
                   0.05 * torch.randn((h, 3), generator=g, device=DEV), _uniform(g, (n - h, 3), -1.0, 1.0)])
    c = torch.stack([0.5 + 0.4 * torch.sin(4 * p[:, 0]), 0.5 + 0.4 * torch.cos(6 * p[:, 1] * p[:, 2]),
                     (p[:, 2] > 0.1) * 0.7 + 0.15], 1) + 0.03 * torch.randn((n, 3), generator=g, device=DEV)
    return p.contiguous(), c.clamp(0, 1).contiguous()


def _particles(case, seed):
    g, k = _gen(seed), case["k"]
    p = torch.zeros((k, 8), device=DEV)
    p[:, 0] = _uniform(g, (k,), 0.0, case["width"])
    p[:, 1] = _uniform(g, (k,), 0.0, case["height"])
    p[:, 2] = _uniform(g, (k,), math.log(1.0), math.log(12.0))
    p[:, 3:6] = torch.rand((k, 3), generator=g, device=DEV) * 0.5
    m = torch.zeros_like(p)
    v = torch.zeros_like(p)
    m[:, :6] = 1e-5 * torch.randn((k, 6), generator=g, device=DEV)
    v[:, :6] = (3e-5 * (0.5 + torch.rand((k, 6), generator=g, device=DEV))) ** 2
    return p, m, v


def _restructure_inputs(case, seed):
    scene = _scene(case, seed, log_params=True)
    m, v = _moments(seed, scene, 1e-6)
    return scene, m, v


# ---------------------------------------------------------- prepare and run --

class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.kind = case, case["kind"]
    return _PREPARE[s.kind](s, case, seed)


def run(state):
    return _RUN[state.kind](state, state.case)


def _prep_render(s, case, seed):
    s.scene = igs.Scene(*_scene(case, seed))
    s.cam = igs.camera(_camera(seed, case["width"], case["height"]))
    s.r = Renderer(tile=case["tile"], sh_degree=case["sh"], device=DEV, footprint=case["footprint"])
    s.img = torch.empty((3, case["height"], case["width"]), device=DEV)
    s.r.run_forward(s.scene, s.cam, img=s.img)  # sizes the frame
    return s


def _run_render(s, case):
    return s.r.run_forward(s.scene, s.cam, img=s.img, check=case["check"])[0]


def _prep_grad(s, case, seed):
    s.params = [t.requires_grad_() for t in _scene(case, seed)]
    s.cam = igs.camera(_camera(seed, case["width"], case["height"]))
    s.dL = _image(seed, case["width"], case["height"], 5) - 0.5
    s.r = Renderer(tile=case["tile"], sh_degree=case["sh"], device=DEV)
    render(*s.params, s.r, s.cam)
    return s


def _run_grad(s, case):
    for t in s.params:
        t.grad = None
    img = render(*s.params, s.r, s.cam)
    img.backward(s.dL)
    return [img] + [t.grad for t in s.params]


def _prep_train(s, case, seed):
    scene = _scene(case, seed, log_params=True)
    m, v = _moments(seed, scene, _train_scale(case))
    s.ts = TrainStep.from_state_dict(dict(
        means_sigma=scene[0], opacity=scene[1], color=scene[2], m=m, v=v, t=TRAIN_T,
        adam_state=torch.tensor([TRAIN_T, 0, 0, 0], dtype=torch.int32), sh_degree=case["sh"], tile=case["tile"],
        lr=TRAIN_LR, fused=True, footprint=0, ssim_lambda=case["ssim"]), device=DEV)
    w, h = case["width"], case["height"]
    s.cams = [igs.camera(_camera(seed, w, h, k)) for k in range(TRAIN_VIEWS)]
    s.targets = [_image(seed, w, h, 10 + k) for k in range(TRAIN_VIEWS)]
    for c in s.cams:  # the entry capacity of every view
        s.ts.renderer.run_forward(s.ts.scene, c)
    s.k = 0
    if case["graph"]:
        s.ts.capture(s.cams, s.targets, chain=True)
    return s


def _run_train(s, case):
    ts = s.ts
    if case["graph"]:
        ts.replay(s.k)
    else:
        ts.step(s.cams[s.k], s.targets[s.k])
    s.k = (s.k + 1) % TRAIN_VIEWS
    return [ts.loss, ts.ms, ts.op, ts.col, list(ts.m_views), list(ts.v_views)]


def _prep_batch(s, case, seed):
    s.scene = igs.Scene(*_scene(case, seed))
    s.br = BatchRenderer(s.scene, _batch_cameras(case, seed), tile=case["tile"], blend_batch=64,
                         sh_degree=case["sh"], device=DEV)
    s.br.capture()
    return s


def _run_batch(s, case):
    s.br.replay()
    return [s.br.image(v) for v in range(case["views"])]


def _prep_serve(s, case, seed):
    s.server = igs.Server(pool_bytes=6 << 30, slots=4, tile=case["tile"], device=DEV)
    s.ids = []
    for k, n in enumerate((case["n"], max(1, case["n"] // 2))):
        s.ids.append(s.server.add_scene(igs.Scene(*_scene(dict(case, n=n), seed + 31 * k)), sh_degree=case["sh"]))
    s.cams = [igs.camera(c) for c in _serve_cameras(case, seed)]
    s.imgs = [torch.empty((3, c.height, c.width), device=DEV) for c in s.cams]
    torch.cuda.synchronize()  # the scenes are resident before the first request
    _run_serve(s, case)       # a server in service has seen these sizes
    return s


def _run_serve(s, case):
    reqs = [s.server.submit(s.ids[k % 2], c, img) for k, (c, img) in enumerate(zip(s.cams, s.imgs))]
    for r in reqs:
        st, _ = s.server.poll(r)
        if st != igs.OK:
            raise RuntimeError(f"request {r}: status {st}")
    return s.imgs


def _prep_fit2d(s, case, seed):
    s.p, s.m, s.v = _particles(case, seed)
    w, h = case["width"], case["height"]
    s.target = _fit_target(case, seed)
    s.img, s.dimg = torch.empty((3, h, w), device=DEV), torch.empty((3, h, w), device=DEV)
    s.grad = torch.zeros_like(s.p)
    s.state = torch.tensor([TRAIN_T, 0], dtype=torch.int32, device=DEV)
    s.loss, s.ssim = torch.zeros(1, device=DEV), torch.zeros(1, device=DEV)
    s.work = torch.empty(igs.ssim_work_bytes(3, h, w) // 4, device=DEV)
    return s


def _run_fit2d(s, case):
    igs.fit2d_render(s.p, case["D"], s.img)
    igs.l1_ssim_loss(s.img, s.target, 0.2, s.loss, s.dimg, s.work, ssim=s.ssim)
    igs.fit2d_backward(s.p, case["D"], s.dimg, s.grad)
    igs.fit2d_adam(s.p, s.grad, s.m, s.v, FIT_LR, s.state)
    return [s.img, s.loss, s.ssim, s.dimg, s.grad, s.p, s.m, s.v]


def _fit_target(case, seed):
    """A smooth image with noise (a photograph's two ingredients)."""
    w, h = case["width"], case["height"]
    x, y = torch.meshgrid(torch.arange(w, device=DEV) / w, torch.arange(h, device=DEV) / h, indexing="xy")
    ph = _uniform(_gen(seed, 6), (3, 1, 1), 0.0, 6.28)
    t = 0.5 + 0.3 * torch.sin(9 * x + ph) * torch.cos(7 * y - ph)
    return (t + 0.05 * torch.randn((3, h, w), generator=_gen(seed, 7), device=DEV)).clamp(0, 1).contiguous()


def _prep_octree(s, case, seed):
    s.points, s.colors = _points(case, seed)
    k, row = case["k_max"], _row(case["sh"]) // 4 - 5
    s.params = [torch.zeros((k, 4), device=DEV), torch.zeros(k, device=DEV), torch.zeros((k, row), device=DEV)]
    return s


def _run_octree(s, case):
    got = igs.octree_init(s.points, s.colors, (-1.0, -1.0, -1.0), 2.0, case["levels"], case["k_max"], opacity=0.5,
                          sh_degree=case["sh"])
    for dst, src in zip(s.params, got):  # into the program's own parameter buffers of k_max Gaussians
        dst[:len(src)].copy_(src)
    return s.params


def _prep_restructure(s, case, seed, capacity, work):
    scene, s.m, s.v = _restructure_inputs(case, seed)
    s.scene = igs.Scene(*scene)
    s.outs = [[torch.zeros((capacity,) + t.shape[1:], device=DEV) for t in scene] for _ in range(3)]
    s.count = torch.zeros(1, dtype=torch.int64, device=DEV)
    s.work = torch.empty(work(case["n"]), dtype=torch.uint8, device=DEV)
    return s


def _prep_merge(s, case, seed):
    return _prep_restructure(s, case, seed, case["n"], igs.merge_work_bytes)


MERGE_SCALE = math.log(0.0158)  # about the median scale of the uniform scene


def _run_merge(s, case):
    igs.merge(s.scene, s.m, s.v, case["sh"], 1, (-1.0, -1.0, -1.0), 2.0 / case["cells"], MERGE_SCALE, *s.outs, s.count,
              s.work)
    return [s.count] + s.outs


def _densify_stats(case, seed):
    g = _gen(seed, 8)
    vis = torch.randint(0, 17, (case["n"],), generator=g, device=DEV, dtype=torch.int32)
    accum = vis * 1e-6 * -torch.log(torch.rand((case["n"],), generator=g, device=DEV).clamp_min(1e-7))
    return accum.contiguous(), vis


DENSIFY = (math.log(0.07 / 0.93), 4e-6, math.log(0.01))  # opacity floor, mean gradient, scale floor


def _densify_capacity(case):
    return case["n"] + case["n"] // 10


def _prep_densify(s, case, seed):
    s.accum, s.vis = _densify_stats(case, seed)
    return _prep_restructure(s, case, seed, _densify_capacity(case), igs.densify_work_bytes)


def _run_densify(s, case):
    igs.densify(s.scene, s.m, s.v, case["sh"], 1, s.accum, s.vis, *DENSIFY, *s.outs, s.count, s.work)
    return [s.count] + s.outs


_PREPARE = dict(render=_prep_render, grad=_prep_grad, train=_prep_train, batch=_prep_batch, serve=_prep_serve,
                fit2d=_prep_fit2d, octree=_prep_octree, merge=_prep_merge, densify=_prep_densify)
_RUN = dict(render=_run_render, grad=_run_grad, train=_run_train, batch=_run_batch, serve=_run_serve,
            fit2d=_run_fit2d, octree=_run_octree, merge=_run_merge, densify=_run_densify)


# -------------------------------------------------------------------- work --

def _row(sh):
    return 4 * (5 + (3 if sh < 0 else 3 * (sh + 1) ** 2))  # bytes of one Gaussian's parameters


def _frame_flops(case, px, focal):
    """Projection and colour of each Gaussian, and about 20 operations for each (pixel, Gaussian) pair inside a
    support radius of three scales, at most 60 layers deep (where a pixel of average opacity stops)."""
    scale = 0.018 if case.get("scene", "uniform") == "uniform" else 0.012
    area = math.pi * (3 * focal * scale / 4) ** 2
    return case["n"] * (80 + 6 * max(1, (case["sh"] + 1) ** 2)) + 20 * min(case["n"] * area, 60 * px)


def work(case):
    kind = case["kind"]
    if kind in ("render", "grad", "train"):
        px = case["width"] * case["height"]
        scene, fl = case["n"] * _row(case["sh"]), _frame_flops(case, px, 0.85 * case["width"])
        if kind == "render":
            return dict(bytes=scene + 12 * px, flops=fl)
        if kind == "grad":  # parameters, image gradient; image, parameter gradients
            return dict(bytes=2 * scene + 24 * px, flops=3 * fl)
        # parameters and both moments read and written, target
        return dict(bytes=6 * scene + 12 * px, flops=3 * fl + 15 * case["n"] * _row(case["sh"]) // 4)
    if kind == "batch":
        sizes = [(c.width, c.height) for c in _batch_cameras(case, 0)]
        return dict(bytes=case["n"] * _row(case["sh"]) + sum(12 * w * h for w, h in sizes),
                    flops=sum(_frame_flops(case, w * h, 0.85 * w) for w, h in sizes))
    if kind == "serve":
        by, fl = 0, 0
        for k, c in enumerate(_serve_cameras(case, 0)):
            one = dict(case, n=case["n"] if k % 2 == 0 else max(1, case["n"] // 2))
            by += one["n"] * _row(case["sh"]) + 12 * c.width * c.height
            fl += _frame_flops(one, c.width * c.height, 0.85 * c.width)
        return dict(bytes=by, flops=fl)
    if kind == "fit2d":
        px = case["width"] * case["height"]
        pairs = case["k"] * min(px, math.pi * case["D"] ** 2)
        return dict(bytes=7 * 32 * case["k"] + 4 * 12 * px, flops=50 * pairs + 3 * px * 250)
    if kind == "octree":
        return dict(bytes=24 * case["n"] + min(case["k_max"], case["n"]) * _row(case["sh"]), flops=20 * case["n"])
    out = case["n"] if kind == "merge" else _densify_capacity(case)
    return dict(bytes=3 * _row(case["sh"]) * (case["n"] + out), flops=20 * case["n"])


# ------------------------------------------------- the same in 64-bit torch --

def exact(case, seed):
    f = _EXACT.get(case["kind"])
    return f(case, seed) if f else None


def _too_big(case):
    return case["n"] * case["width"] * case["height"] > EXACT_PAIRS


def _sh_basis(deg, d):
    """Real spherical harmonics (no Condon-Shortley phase) of unit directions [n,3], index l^2 + l + m."""
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        a = math.sqrt(3 / (4 * math.pi))
        Y += [a * y, a * z, a * x]
    if deg >= 2:
        a = 0.5 * math.sqrt(15 / math.pi)
        Y += [a * x * y, a * y * z, 0.25 * math.sqrt(5 / math.pi) * (3 * z * z - 1), a * x * z,
              0.5 * a * (x * x - y * y)]
    if deg >= 3:
        a, b, c = 0.25 * math.sqrt(35 / (2 * math.pi)), 0.5 * math.sqrt(105 / math.pi), 0.25 * math.sqrt(21 / (2 * math.pi))
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1),
              0.25 * math.sqrt(7 / math.pi) * z * (5 * z * z - 3), c * x * (5 * z * z - 1), 0.5 * b * z * (x * x - y * y),
              a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _project64(ms, op, col, sh, cam):
    """Discs (u, v, 1 / (2 s^2), opacity, rgb) of the Gaussians before the camera, front to back."""
    R, t = torch.tensor(cam.R, dtype=torch.float64, device=DEV), torch.tensor(cam.t, dtype=torch.float64, device=DEV)
    x = ms[:, :3] @ R.T + t
    with torch.no_grad():
        keep = torch.nonzero((x[:, 2] > cam.znear) & (ms[:, 3] > 0) & (op >= 1 / 255))[:, 0]
        keep = keep[torch.sort(x[keep, 2].float(), stable=True).indices]
    x, sg, o, c = x[keep], ms[keep, 3], op[keep], col[keep]
    u, v, sc = cam.fx * x[:, 0] / x[:, 2] + cam.cx, cam.fy * x[:, 1] / x[:, 2] + cam.cy, cam.fx * sg / x[:, 2]
    if sh >= 0:
        d = torch.nn.functional.normalize(ms[keep, :3] + R.T @ t, dim=1)
        c = ((_sh_basis(sh, d)[:, :, None] * c.view(len(c), -1, 3)).sum(1) + 0.5).clamp_min(0)
    return u, v, 0.5 / (sc * sc), o, c


def _blend64(disc, px, py):
    """Front-to-back compositing of the pixels: alpha = min(0.99, o exp(-d^2 / 2 s^2)), skipped below 1/255,
    stopped before the transmittance falls below 1e-4. Returns [3, pixels]."""
    u, v, w, o, c = disc
    d2 = (px[:, None] - u) ** 2 + (py[:, None] - v) ** 2
    a = torch.clamp_max(o * torch.exp(-d2 * w), 0.99)
    a = torch.where(a >= 1 / 255, a, torch.zeros_like(a))
    after = torch.cumprod(1 - a, 1)
    before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
    return (torch.where(after >= 1e-4, a * before, torch.zeros_like(a)) @ c).T


def _render64(case, params, cam, dL=None):
    """The image [3,H,W] in 64 bits; with dL (or a function of the image that gives it) the gradients too."""
    w, h, sh = case["width"], case["height"], case["sh"]
    yy, xx = torch.meshgrid(torch.arange(h, device=DEV) + 0.5, torch.arange(w, device=DEV) + 0.5, indexing="ij")
    px, py = xx.reshape(-1).double(), yy.reshape(-1).double()
    step = max(1, int(4e7 // max(1, case["n"])))
    with torch.no_grad():
        disc = _project64(*params, sh, cam)
        img = torch.cat([_blend64(disc, px[i:i + step], py[i:i + step]) for i in range(0, w * h, step)], 1)
        img = img.view(3, h, w)
    if dL is None:
        return img
    dL = dL(img) if callable(dL) else dL
    leaves = [t.detach().requires_grad_() for t in params]
    disc = _project64(*leaves, sh, cam)
    cut = [t.detach().requires_grad_() for t in disc]
    flat = dL.reshape(3, -1)
    for i in range(0, w * h, step):
        (_blend64(cut, px[i:i + step], py[i:i + step]) * flat[:, i:i + step]).sum().backward()
    torch.autograd.backward([t for t in disc if t.requires_grad], [q.grad for q, t in zip(cut, disc) if t.requires_grad])
    return img, [t.grad for t in leaves]


def _double(ts):
    return [t.double() for t in ts]


def _exact_render(case, seed):
    if _too_big(case):
        return None
    return _render64(case, _double(_scene(case, seed)), _camera(seed, case["width"], case["height"]))


def _exact_grad(case, seed):
    if _too_big(case):
        return None
    dL = (_image(seed, case["width"], case["height"], 5) - 0.5).double()
    img, grads = _render64(case, _double(_scene(case, seed)), _camera(seed, case["width"], case["height"]), dL)
    return [img] + grads


def _loss64(img, target, lam):
    """(1 - lam) L1 + lam (1 - SSIM), its image gradient, and the SSIM (11 x 11 Gaussian window, zeros outside)."""
    x = img.detach().requires_grad_()
    k = torch.exp(-(torch.arange(-5, 6, device=DEV).double() ** 2) / 4.5)
    k = (k / k.sum())
    win = (k[:, None] * k)[None, None]

    def mean(a):
        return torch.nn.functional.conv2d(a[:, None], win, padding=5)[:, 0]
    mx, my = mean(x), mean(target)
    sxx, syy, sxy = mean(x * x) - mx * mx, mean(target * target) - my * my, mean(x * target) - mx * my
    ssim = ((2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sxx + syy + 9e-4))).mean()
    loss = (1 - lam) * (x - target).abs().mean() + lam * (1 - ssim)
    loss.backward()
    return loss.detach(), x.grad, ssim.detach()


def _adam64(p, g, m, v, t, lr):
    m, v = 0.9 * m + (1 - 0.9) * g, 0.999 * v + (1 - 0.999) * g * g
    return p - lr / (1 - 0.9 ** t) * m / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8), m, v


def _exact_train(case, seed):
    if _too_big(case):
        return None
    stored = _scene(case, seed, log_params=True)
    mm, vv = _moments(seed, stored, _train_scale(case))
    p = _double(stored)
    sigma, o = torch.exp(p[0][:, 3]), torch.sigmoid(p[1])
    linear = [torch.cat([p[0][:, :3], sigma[:, None]], 1), o, p[2]]
    target, got = _image(seed, case["width"], case["height"], 10).double(), {}

    def dL(img):
        got["loss"], g, _ = _loss64(img, target, case["ssim"])
        return g
    _, g = _render64(case, linear, _camera(seed, case["width"], case["height"]), dL)
    g[0][:, 3] *= sigma
    g[1] *= o * (1 - o)
    new = [_adam64(a, b, m, v, TRAIN_T + 1, TRAIN_LR) for a, b, m, v in zip(p, g, _double(mm), _double(vv))]
    return [got["loss"].reshape(1)] + [x[0] for x in new] + [[x[1] for x in new], [x[2] for x in new]]


def _exact_fit2d(case, seed):
    w, h, D = case["width"], case["height"], case["D"]
    p, m, v = _double(_particles(case, seed))
    yy, xx = torch.meshgrid(torch.arange(h, device=DEV) + 0.5, torch.arange(w, device=DEV) + 0.5, indexing="ij")
    px, py = xx.reshape(-1).double(), yy.reshape(-1).double()
    near = p.float()

    def kernel(q, i, j):
        # which pairs are reached is decided in 32 bits, as the path defines it
        fx, fy = px[i:j].float()[:, None] - near[:, 0], py[i:j].float()[:, None] - near[:, 1]
        reach = fx * fx + fy * fy < torch.tensor(D, device=DEV).float() ** 2
        d2 = (px[i:j, None] - q[:, 0]) ** 2 + (py[i:j, None] - q[:, 1]) ** 2
        g = torch.exp(-d2 * 0.5 * torch.exp(-2 * q[:, 2]))
        return (torch.where(reach, g, torch.zeros_like(g)) @ q[:, 3:6]).T
    step = max(1, int(4e7 // case["k"]))
    with torch.no_grad():
        img = torch.cat([kernel(p, i, i + step) for i in range(0, w * h, step)], 1).view(3, h, w)
    loss, dimg, ssim = _loss64(img, _fit_target(case, seed).double(), 0.2)
    q, flat = p.detach().requires_grad_(), dimg.reshape(3, -1)
    for i in range(0, w * h, step):
        (kernel(q, i, i + step) * flat[:, i:i + step]).sum().backward()
    new = _adam64(p, q.grad, m, v, TRAIN_T + 1, torch.tensor(FIT_LR, device=DEV).double())
    return [img, loss.reshape(1), ssim.reshape(1), dimg, q.grad, *new]


def _exact_octree(case, seed):
    """The greedy tree as a prefix of the cells in (error descending, id ascending) order."""
    pts, cols = _points(case, seed)
    L, n = case["levels"], case["n"]
    ix = torch.floor((pts + 1.0) * (2.0 ** L / 2.0)).clamp(0, 2 ** L - 1).long()
    cell = torch.zeros(n, dtype=torch.int64, device=DEV)
    for b in range(L):
        for a in range(3):
            cell |= ((ix[:, a] >> b) & 1) << (3 * b + a)
    q = torch.round(cols.clamp(0, 1) * 4096).long()
    stats = torch.zeros((8 ** L, 7), dtype=torch.int64, device=DEV)
    stats.index_add_(0, cell, torch.cat([torch.ones((n, 1), dtype=torch.int64, device=DEV), q, q * q], 1))
    levels = [stats]
    for _ in range(L):
        levels.insert(0, levels[0].view(-1, 8, 7).sum(1))
    key, inc, ids, off = [], [], [], 0
    for lv in range(L):
        s = levels[lv].double()
        e = torch.zeros(len(s), dtype=torch.float64, device=DEV)
        for c in range(3):
            e = e + (s[:, 4 + c] - s[:, 1 + c] * s[:, 1 + c] / s[:, 0].clamp_min(1))
        e = e.clamp_min(0)
        key.append(e if lv == 0 else torch.minimum(e, key[-1].repeat_interleave(8)))
        kids = (levels[lv + 1][:, 0] > 0).view(-1, 8).sum(1) - 1
        inc.append(torch.where(levels[lv][:, 0] >= 2, kids, torch.full_like(kids, -1)))
        ids.append(off + torch.arange(len(s), device=DEV))
        off += len(s)
    key, inc, ids = torch.cat(key), torch.cat(inc), torch.cat(ids)
    ok = inc >= 0
    order = ids[ok][torch.sort(key[ok], descending=True, stable=True).indices]
    fits = 1 + torch.cumsum(inc[order], 0) <= case["k_max"]
    split = torch.zeros(off, dtype=torch.bool, device=DEV)
    split[order[: int(fits.sum()) if not fits.all() else len(order)]] = True
    out, at = [], 0
    for lv in range(L + 1):
        s, k = levels[lv], 8 ** lv
        leaf = s[:, 0] > 0
        if lv > 0:
            leaf &= split[at - k // 8:at].repeat_interleave(8)
        if lv < L:
            leaf &= ~split[at:at + k]
        mor = torch.nonzero(leaf)[:, 0]
        pos = torch.zeros((len(mor), 3), dtype=torch.float64, device=DEV)
        for b in range(lv):
            for a in range(3):
                pos[:, a] += ((mor >> (3 * b + a)) & 1) << b
        side = 2.0 / 2 ** lv
        mean = s[mor, 1:4].double() / (4096.0 * s[mor, :1].double())
        out.append((torch.cat([-1.0 + (pos + 0.5) * side, torch.full((len(mor), 1), side / 2, device=DEV).double()], 1),
                    mean))
        at += k
    ms, mean = torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])
    if case["sh"] >= 0:
        col = torch.zeros((len(ms), 3 * (case["sh"] + 1) ** 2), dtype=torch.float64, device=DEV)
        col[:, :3] = (mean - 0.5) * 2 * math.sqrt(math.pi)
        mean = col
    op = torch.full((len(ms),), 0.5, dtype=torch.float64, device=DEV)
    return [_pad(t, case["k_max"]) for t in (ms, op, mean)]


def _pad(rows, capacity):
    return torch.cat([rows, torch.zeros((capacity - len(rows),) + rows.shape[1:], dtype=rows.dtype, device=DEV)])


def _exact_merge(case, seed):
    scene, m, v = _restructure_inputs(case, seed)
    n = case["n"]
    inv = (1.0 / torch.tensor(2.0 / case["cells"], dtype=torch.float32)).item()
    c = torch.floor((scene[0][:, :3] - (-1.0)) * inv).long()
    ok = (scene[0][:, 3] <= torch.tensor(MERGE_SCALE).float().item()) & ((c >= 0) & (c < 1024)).all(1)
    key = torch.where(ok, c[:, 0] | (c[:, 1] << 10) | (c[:, 2] << 20), torch.arange(n, device=DEV) + (1 << 40))
    _, group, size = torch.unique(key, return_inverse=True, return_counts=True)
    idx = torch.arange(n, device=DEV)
    first = torch.full((len(size),), n, dtype=torch.int64, device=DEV).scatter_reduce(0, group, idx, "amin")
    lead = first[group] == idx
    ms, op, col = _double(scene)
    o, sg = torch.sigmoid(op), torch.exp(ms[:, 3])

    def total(x):
        return torch.zeros((len(size),) + x.shape[1:], dtype=torch.float64, device=DEV).index_add_(0, group, x)
    W = total(o)
    mu = total(o[:, None] * ms[:, :3]) / W[:, None]
    var = total(o * (sg * sg + ((ms[:, :3] - mu[group]) ** 2).sum(1) / 3)) / W
    log_keep = total(-torch.nn.functional.softplus(op))
    cover = -torch.expm1(log_keep)
    logit = torch.where(cover >= 0.99, torch.full_like(cover, math.log(99.0)), torch.log(cover) - log_keep)
    merged = (size > 1)[group][lead]
    g = group[lead]
    new = [torch.cat([mu, 0.5 * torch.log(var)[:, None]], 1), logit, total(o[:, None] * col) / W[:, None]]

    def pick(old, rows):
        return torch.where(merged.view((-1,) + (1,) * (old.dim() - 1)), rows, old)
    out = [[pick(a[lead], b[g]) for a, b in zip((ms, op, col), new)]]
    out += [[pick(a[lead], torch.zeros_like(a[lead])) for a in _double(mom)] for mom in (m, v)]
    return [None] + [[_pad(t, n) for t in block] for block in out]


def _exact_densify(case, seed):
    scene, m, v = _restructure_inputs(case, seed)
    accum, vis = _densify_stats(case, seed)
    cap = _densify_capacity(case)
    op_min, tau, smin = (torch.tensor(x).float().item() for x in DENSIFY)
    keep = ~(scene[1] < op_min)
    cand = keep & (vis > 0) & (accum > torch.tensor(tau, device=DEV).float() * vis.float()) & (scene[0][:, 3] >= smin)
    divide = cand & (torch.cumsum(cand, 0) <= max(0, cap - int(keep.sum())) // 7)
    rep = torch.where(divide, 8, keep.long())
    src = torch.repeat_interleave(torch.arange(case["n"], device=DEV), rep)
    child = torch.arange(len(src), device=DEV) - (torch.cumsum(rep, 0) - rep)[src]
    d = divide[src]
    src, child, d = src[:cap], child[:cap], d[:cap]
    ms, op, col = (t[src] for t in _double(scene))
    sign = torch.stack([((child >> a) & 1) * 2.0 - 1.0 for a in range(3)], 1).double()
    moved = torch.cat([ms[:, :3] + 0.5 * torch.exp(ms[:, 3:]) * sign, ms[:, 3:] - math.log(2.0)], 1)
    ms = torch.where(d[:, None], moved, ms)
    out = [[ms, op, col]]
    for mom in (m, v):
        out.append([torch.where(d.view((-1,) + (1,) * (t.dim() - 1)), torch.zeros_like(t[src]).double(),
                                t[src].double()) for t in mom])
    return [None] + [[_pad(t, cap) for t in block] for block in out]


_EXACT = dict(render=_exact_render, grad=_exact_grad, train=_exact_train, fit2d=_exact_fit2d, octree=_exact_octree,
              merge=_exact_merge, densify=_exact_densify)
