"""Calls of one context one after another, where the culling's counts and the connection
weights' error flag reach the host: every call reports its own eyes only, whatever the call
before it was (fewer blocks, more, none, an overflow, an error). Counts are whole numbers, equal
to the oracle's."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import oracle_hier, upload_scene
from test_gpu_connect import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lights", [1, 5003])
def test_each_call_reports_its_own(ctx, lights):  # noqa: F811
    import torch
    import paper_1907_12343_gb300 as hrr
    s = dict(synth.scene_frame(width=61, height=37, n_lights=5003, tile_w=16, tile_h=16, target=24.0, seed=5))
    s["light_pos"], s["intensity"] = s["light_pos"][:lights], s["intensity"][:lights]
    g = upload_scene(s)
    e, l = [g[k] for k in ("ex", "ey", "ez", "px", "py")], [g[k] for k in ("lx", "ly", "lz", "li")]
    ctx.set_shift_tile(s["tile"])
    tree = ctx.build_light_tree(*l)
    tau, n_e = float(s["tau"]) * 5003 / lights, len(s["eye_pos"])
    want = oracle_hier(oracle.Tree(s["light_pos"], s["intensity"]), s["eye_pos"], s["px"], s["py"], s["tile"],
                       np.float32(tau))
    per_eye = np.bincount(want["pairs"][:, 0].astype(np.int64), minlength=n_e)
    pairs = torch.empty((int(per_eye.sum()) + 8, 2), dtype=torch.int32, device=e[0].device)
    sums = torch.empty(n_e, device=e[0].device)
    for n in (1, n_e, 0, 9, 8, n_e, 33):
        part = [a[:n] for a in e]
        st, cnt = ctx.cull(*part, tree, tau, pairs)
        assert (st, cnt) == (hrr.HRR_OK, int(per_eye[:n].sum()))
        assert ctx.last_cull_stats() == (int(want["visits"][:n].sum()), cnt)
        if n == n_e and cnt > 1:
            assert ctx.cull(*part, tree, tau, pairs[:1]) == (hrr.HRR_ERR_OVERFLOW, cnt)
            ctx.cull(*part, tree, tau, pairs)
        if cnt:
            bad = pairs.clone()
            bad[cnt // 2, 1] = lights
            for p, ok in ((pairs, True), (bad, False), (pairs, True)):
                if ok:
                    ctx.connect(*part[:3], tuple(l), tau, p, cnt, eye_sum=sums)
                else:
                    with pytest.raises(Exception):
                        ctx.connect(*part[:3], tuple(l), tau, p, cnt, eye_sum=sums)
    tree.free()
