"""The build's sort and box pass at the sizes and keys where they change path: tiles of 1024
and 4096 keys and the switch between them at 2^17 lights, box blocks of 512 leaves, groups of
32^k, and runs of lights that share the upper half of their keys, up to and past the longest
run put in order without a full sort (64). Trees equal the oracle's node by node."""
import numpy as np
import pytest

from test_gpu_build import _compare, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def _runs(rng, n, length):
    """n lights in groups of `length` whose keys agree in the upper 32 of 63 bits, shuffled."""
    groups = -(-n // length)
    cell = rng.integers(0, 1 << 10, size=(groups, 3)) << 11  # the upper bits of each axis
    pos = np.repeat(cell, length, axis=0)[:n] + rng.integers(0, 1 << 10, size=(n, 3))
    return (rng.permutation(pos) / 2.0 ** 21).astype(np.float32)


@pytest.mark.parametrize("n", [31, 65, 511, 512, 513, 1024, 1025, 2049, 16385, 131072, 131073, 135169])
def test_sizes_at_tile_and_block_edges(ctx, n):  # noqa: F811
    rng = np.random.default_rng(n)
    _compare(ctx, rng.random((n, 3)).astype(np.float32), np.exp(rng.standard_normal(n)).astype(np.float32))


@pytest.mark.parametrize("n, length", [(3000, 2), (3000, 63), (3000, 64), (3000, 65), (3000, 3000), (140000, 64),
                                       (140000, 140000)])
def test_runs_of_equal_upper_halves(ctx, n, length):  # noqa: F811
    rng = np.random.default_rng(n + length)
    _compare(ctx, _runs(rng, n, length), np.exp(rng.standard_normal(n)).astype(np.float32))


@pytest.mark.parametrize("n", [300, 5000])
def test_equal_positions_keep_their_order(ctx, n):  # noqa: F811
    pos = np.full((n, 3), 0.3, np.float32)
    pos[n // 2:] = 0.7
    _compare(ctx, pos, np.arange(1, n + 1, dtype=np.float32))
