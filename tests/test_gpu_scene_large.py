"""Shadow segments with a zero (or nearly zero) component through nodes so large that the slab
arithmetic leaves the range of float32: an occluder around such a segment still blocks it.
Visibility is bit-exact against the oracle's brute force over every triangle."""
import numpy as np
import pytest

import oracle
from gpu_util import dev
from test_gpu_connect import ctx  # noqa: F401

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.mark.parametrize("n, size", [(2, 3e7), (2, 9e7), (2, 1.2e8), (2, 2e8), (2, 1e9), (2, 1e12), (9, 1.2e8), (300, 9e7),
                                     (300, 1.2e8), (300, 3e5), (300, 1e10)])
@pytest.mark.parametrize("small", [0.0, 1e-28])
def test_axis_aligned_segments_in_large_nodes(ctx, n, size, small):  # noqa: F811
    import torch
    rng = np.random.default_rng(n)
    tris = rng.uniform(-1, 1, (n, 1, 3)) + 0.2 * rng.uniform(-1, 1, (n, 3, 3))
    for k in range(min(n, 3)):  # sheets across axis k
        tris[k] = [[-1, -1, -1], [3, -1, -1], [-1, 3, -1]]
        tris[k, :, 2] = 0.1 * k
        tris[k] = np.roll(tris[k], k, axis=1)
    tris = (size * tris).astype(F)
    tris[0, :, 2] = 0.0
    if n > 2:
        tris[2] = [[400 * size, 0, 0], [-400 * size, 1, 0], [0, 0, 400 * size]]  # and one far larger than the rest
    n_s = 900
    eyes = (size * rng.uniform(-0.5, 0.5, (n_s, 3))).astype(F)
    lights = eyes.copy()
    axis = rng.integers(0, 3, n_s)
    length = size * 10.0 ** rng.uniform(-3, 1, n_s) * np.where(rng.random(n_s) < 0.5, -1, 1)
    eyes[np.arange(n_s), axis] = lights[np.arange(n_s), axis] = 0
    eyes[np.arange(n_s), axis] -= (0.4 * length).astype(F)
    lights[np.arange(n_s), axis] += (0.6 * length).astype(F)
    eyes[:n_s // 3, 2] -= F(0.25 * size)  # two components
    k = np.arange(2 * n_s // 3, n_s)  # a nearly zero one
    eyes[k, (axis[k] + 1) % 3], lights[k, (axis[k] + 1) % 3] = 0, small
    pairs = np.stack([np.arange(n_s), np.arange(n_s)], 1).astype(np.uint32)
    inten = np.ones(n_s, F)
    t = [torch.from_numpy(np.ascontiguousarray(a)).to(dev()) for a in (*eyes.T, *lights.T, inten, tris.reshape(n, 9))]
    scene = ctx.build_scene(t[7])
    v = torch.zeros(n_s, dtype=torch.uint8, device=dev())
    ctx.connect(*t[:3], tuple(t[3:7]), 1e-3, torch.from_numpy(pairs.view(np.int32)).to(dev()), n_s, scene=scene, visible=v,
                eye_sum=torch.zeros(n_s, device=dev()))
    scene.free()
    want = oracle.connect(eyes, lights, inten, pairs, F(1e-3), tris.reshape(n, 9))["visible"]
    assert 0 < want.sum() < n_s  # both answers occur
    assert np.array_equal(v.cpu().numpy().astype(bool), want)
