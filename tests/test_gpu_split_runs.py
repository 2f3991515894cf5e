"""Cost-driven builds of lights whose keys agree in their upper halves in runs too long to be put
in order without a full sort (the build then starts over): below and above 1024 lights, with
ranges that the cost splits, the radix rule or both take. Splits equal the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import upload_scene
from test_gpu_build import ctx  # noqa: F401
from test_gpu_sort import _runs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, length", [(65, 65), (100, 100), (700, 70), (1024, 1024), (1025, 300), (5000, 5000), (40000, 900)])
@pytest.mark.parametrize("depth", [0, 1, 3])
def test_splits_after_a_full_sort(ctx, n, length, depth):  # noqa: F811
    rng = np.random.default_rng(n + depth)
    pos = _runs(rng, n, length)
    inten = np.exp(1.5 * rng.standard_normal(n)).astype(np.float32)
    g = upload_scene({"light_pos": pos, "intensity": inten, "eye_pos": pos[:1], "px": np.zeros(1, np.uint16),
                      "py": np.zeros(1, np.uint16)})
    tree = ctx.build_light_tree(g["lx"], g["ly"], g["lz"], g["li"], topology="cost", cost_depth=depth)
    nodes, perm = tree.download()
    t = oracle.Tree(pos, inten, topology="cost", **({"cost_depth": depth} if depth else {}))
    assert np.array_equal(perm, t.perm) and tree.height == t.height
    assert np.array_equal(nodes["split"], t.split)
    tree.free()
