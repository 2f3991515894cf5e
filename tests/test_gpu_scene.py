"""Scenes whose nodes hold quantised boxes, where the quantisation and the tree's shape can go
wrong: few triangles (partly filled nodes), sizes around whole levels, scenes far from the origin,
tiny and huge ones, flat ones, and triangles that share one centroid. Visibility and weights are
bit-exact against the oracle's brute force over every triangle."""
import numpy as np
import pytest

import oracle
from gpu_util import dev
from test_gpu_connect import ctx  # noqa: F401

pytestmark = pytest.mark.gpu
F = np.float32


def _triangles(rng, n, kind):
    c = rng.random((n, 1, 3))
    off = 0.15 * n ** (-1 / 3) * rng.standard_normal((n, 3, 3))
    if kind == "flat":
        off[:, :, 2] = 0.0
        c[:, :, 2] = 0.5
    if kind == "same":
        c[:] = 0.5
        off = 0.3 * rng.standard_normal((n, 3, 3))
        off -= off.mean(axis=1, keepdims=True)
    return c + off


@pytest.mark.parametrize("n, kind, scale, shift", [(2, "", 1, 0), (3, "", 1, 0), (8, "", 1, 0), (9, "", 1, 0), (64, "", 1, 0),
                                                   (65, "", 1, 0), (513, "", 1, 0), (4000, "", 1, 0), (700, "flat", 1, 0),
                                                   (300, "same", 1, 0), (1500, "", 1, 1000), (1500, "", 1e-4, 0),
                                                   (1500, "", 1e6, -3e6), (200, "", 1e30, 0)])
def test_visibility_equals_brute_force(ctx, n, kind, scale, shift):  # noqa: F811
    import torch
    rng = np.random.default_rng(n)
    n_e, n_l, n_p = 60, 500, 3000
    place = lambda x: (x * scale + shift).astype(F)  # noqa: E731
    tris = place(_triangles(rng, n, kind)).reshape(n, 9)
    eyes, lights = place(rng.random((n_e, 3)) * 1.2 - 0.1), place(rng.random((n_l, 3)) * 1.2 - 0.1)
    lights[:40, 0] = eyes[0, 0]  # segments with a zero component
    lights[40:60] = eyes[1]      # and of no length
    inten = np.ones(n_l, F)
    pairs = np.stack([rng.integers(0, n_e, n_p), rng.integers(0, n_l, n_p)], 1).astype(np.uint32)
    pairs[:60, 0], pairs[:60, 1] = [0] * 40 + [1] * 20, np.arange(60)
    tau = F(1e-3)
    t = [torch.from_numpy(np.ascontiguousarray(a)).to(dev()) for a in (*eyes.T, *lights.T, inten, tris)]
    scene = ctx.build_scene(t[7])
    w = torch.zeros(n_p, device=dev())
    v = torch.zeros(n_p, dtype=torch.uint8, device=dev())
    s = torch.zeros(n_e, device=dev())
    ctx.connect(*t[:3], tuple(t[3:7]), float(tau), torch.from_numpy(pairs.view(np.int32)).to(dev()), n_p, scene=scene,
                weight=w, visible=v, eye_sum=s)
    want = oracle.connect(eyes, lights, inten, pairs, tau, tris)
    assert np.array_equal(v.cpu().numpy().astype(bool), want["visible"])
    got = w.cpu().numpy()
    nan = np.isnan(want["weight"])  # at the largest scale d^2 overflows; a NaN's bits are the machine's
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint32), want["weight"][~nan].view(np.uint32))
    scene.free()
