"""The cost-driven topology at the sizes where its kernels change: subtrees of up to 32, 64, 128,
256 and 1024 lights, two tiles and more, and cost depths that hand ranges of every size to the
radix rule. Splits equal the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import upload_scene
from test_gpu_build import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, depth", [(2, 0), (32, 0), (33, 0), (64, 0), (65, 0), (128, 0), (129, 0), (256, 0), (257, 0),
                                      (1024, 0), (1025, 0), (2049, 0), (40000, 0), (33, 1), (1024, 2), (1025, 1),
                                      (40000, 1), (40000, 6), (40000, 12)])
def test_splits_equal_the_oracle(ctx, n, depth):  # noqa: F811
    rng = np.random.default_rng(n + depth)
    pos = (rng.random((n, 3)) ** 2).astype(np.float32)
    inten = np.exp(1.5 * rng.standard_normal(n)).astype(np.float32)
    g = upload_scene({"light_pos": pos, "intensity": inten, "eye_pos": pos[:1], "px": np.zeros(1, np.uint16),
                      "py": np.zeros(1, np.uint16)})
    tree = ctx.build_light_tree(g["lx"], g["ly"], g["lz"], g["li"], topology="cost", cost_depth=depth)
    nodes, perm = tree.download()
    t = oracle.Tree(pos, inten, topology="cost", **({"cost_depth": depth} if depth else {}))
    assert np.array_equal(perm, t.perm) and tree.height == t.height
    assert np.array_equal(nodes["split"], t.split)
    tree.free()
