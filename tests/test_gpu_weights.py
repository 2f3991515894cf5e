"""Connection weights without a scene where the kernel's path changes: runs of one eye's pairs of
every length around a warp, eyes that come back within a warp, ragged ends, and both ways to read
the lights (packed from 2^20 pairs on). Weights are bit-exact against the oracle; per-eye sums
within (n + 1) 2^-23 relative, n float32 additions in any order."""
import numpy as np
import pytest

import oracle
from gpu_util import dev
from test_gpu_connect import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, run", [(1, 1), (31, 40), (33, 2), (127, 31), (129, 32), (4097, 33), (1000, 0),
                                    ((1 << 20) - 1, 30), ((1 << 20) + 77, 30), ((1 << 20) + 77, 0)])
def test_runs_of_pairs(ctx, n, run):  # noqa: F811
    import torch
    rng = np.random.default_rng(n + run)
    n_e, n_l = 700, 5003
    eye_pos, light_pos = (rng.random((m, 3)).astype(np.float32) for m in (n_e, n_l))
    inten = np.exp(rng.standard_normal(n_l)).astype(np.float32)
    tau = np.float32(1e-3)
    eyes = np.repeat(rng.integers(0, n_e, n // run + 1), run)[:n] if run else rng.integers(0, 2, n)  # 0: two eyes, mixed
    pairs = np.stack([eyes, rng.integers(0, n_l, n)], 1).astype(np.uint32)
    t = [torch.from_numpy(np.ascontiguousarray(a)).to(dev()) for a in (*eye_pos.T, *light_pos.T, inten)]
    dp = torch.from_numpy(pairs.view(np.int32)).to(dev())
    w = torch.full((n + 1,), -1.0, device=dev())
    v = torch.full((n + 1,), 7, dtype=torch.uint8, device=dev())
    s = torch.full((n_e,), -1.0, device=dev())
    ctx.connect(*t[:3], tuple(t[3:]), float(tau), dp, n, weight=w, visible=v, eye_sum=s)
    want = oracle.connect(eye_pos, light_pos, inten, pairs, tau, None)
    assert np.array_equal(w[:n].cpu().numpy().view(np.uint32), want["weight"].view(np.uint32))
    assert float(w[n]) == -1.0 and bool((v[:n] == 1).all()) and int(v[n]) == 7
    per_eye = np.bincount(pairs[:, 0].astype(np.int64), minlength=n_e)
    exact = np.bincount(pairs[:, 0].astype(np.int64), weights=want["weight"].astype(np.float64), minlength=n_e)
    assert np.all(np.abs(s.cpu().numpy() - exact) <= (per_eye + 1) * 2.0 ** -23 * exact + 1e-30)
