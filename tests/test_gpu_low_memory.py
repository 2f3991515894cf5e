"""Builds where the memory of the context's pool ends (a stand-in for the runtime's allocation
refuses): with too little for the hierarchy itself HRR_ERR_OOM, and nothing kept; with room for all
but the paired records a hierarchy that gives every call the same pairs and visits as one with
them."""
import pytest

import fake_lib

pytestmark = pytest.mark.gpu

HEAD = """
import os
import numpy as np, torch
import paper_1907_12343_gb300 as hrr
import synth
from gpu_util import dev, run_cull, sorted_pairs, upload_scene
assert hrr.__file__.startswith(os.getcwd())
used = hrr._lib.hrr_fake_used
used.restype = hrr._u64
ctx = hrr.Context(0)
"""

LIGHTS = HEAD + """
s = dict(synth.scene_frame(width=61, height=37, n_lights=40000, tile_w=16, tile_h=16, target=24.0, seed=5))
n_e, cap = len(s["eye_pos"]), 1 << 18
tile = torch.from_numpy(np.ascontiguousarray(s["tile"]).view(np.int32)).to(dev())
ctx.set_shift_tile(s["tile"])
kept = used()

def results(g, tree, tau, lights):
    out = []
    for t in ({}, {"top_levels": 1}, {"rangemin_variant": 2}, {"threads_per_block": 128, "ring_entries": 128}, {"node_width": 4}):
        st, cnt, pairs, vis = run_cull(ctx, g, tree, tau, cap=cap, visits=True, tuning=t)
        assert st == hrr.HRR_OK
        out += [sorted_pairs(pairs), vis]
    e = [g[k] for k in ("ex", "ey", "ez", "px", "py")]
    p = torch.empty((3, cap, 2), dtype=torch.int32, device=dev())
    st, counts, visits = ctx.cull_samples(*e, tree, tau, [0, 1 << 31, 12345], p)
    assert st == hrr.HRR_OK
    out += [sorted_pairs(p[k, :c].cpu().numpy().view(np.uint32)) for k, c in enumerate(counts)] + [np.array(visits)]
    host = torch.empty((cap, 2), dtype=torch.int32)
    st, cnt = ctx.cull_host(*[a.cpu() for a in e], tree, tau, host)
    out.append(sorted_pairs(host[:cnt].numpy().view(np.uint32)))
    return out

def together(g, trees, tau):  # frames of both kinds in one batch, jobs of both in one slice
    names = ("x", "y", "z", "px", "py")
    e = [g[k] for k in ("ex", "ey", "ez", "px", "py")]
    frames = [dict(zip(names, e), tree=t, tau=tau, tile=tile, pairs=torch.empty((cap, 2), dtype=torch.int32, device=dev()))
              for t in trees]
    b = hrr.Batch(ctx, frames)
    b.launch()
    st, counts, visits = b.results()
    out = [[sorted_pairs(f["pairs"][:c].cpu().numpy().view(np.uint32)), np.array(v)] for f, c, v in zip(frames, counts, visits)]
    b.destroy()
    srv = hrr.Server(ctx, hbm_budget_bytes=1 << 30)
    tickets = [srv.submit(*e, t, tau, cap, tile=tile) for t in trees]
    for t, o in zip(tickets, out):
        r = srv.wait(t, 60.0)
        assert r["status"] == hrr.HRR_OK
        o += [sorted_pairs(srv.pairs(t, r)), np.array(r["visits"])]
        srv.release(t)
    srv.destroy()
    return out

def same(a, b):
    assert len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))

for n, topology in ((1, "radix"), (2, "radix"), (2, "cost"), (33, "cost"), (700, "radix"), (5000, "cost"), (40000, "cost"),
                    (40000, "radix")):
    part = dict(s, light_pos=s["light_pos"][:n], intensity=s["intensity"][:n])
    g, tau = upload_scene(part), float(s["tau"]) * 40000 / n
    l = [g[k] for k in ("lx", "ly", "lz", "li")]
    whole = ctx.build_light_tree(*l, topology=topology)
    size = used() - kept
    assert size >= 324 * (n - 1)
    want = results(g, whole, tau, l)
    refused, most = 0, size // 8
    while True:  # the least memory that suffices
        os.environ["HRR_FAKE_MEMORY"] = str(kept + size + most)
        try:
            tree = ctx.build_light_tree(*l, topology=topology)
            break
        except hrr.HRRError as e:
            assert e.status == hrr.HRR_ERR_OOM, e
            assert used() == kept + size
            refused += 1
            most += max(32, size // 64)
    del os.environ["HRR_FAKE_MEMORY"]
    bare = used() - kept - size
    assert refused and bare == size - 128 * max(n - 1, 1), (refused, bare, size)
    assert bare <= 196 * n + 4096
    a, b = whole.download(), tree.download()
    assert tree.height == whole.height and all(x.tobytes() == y.tobytes() for x, y in zip(a, b))
    same(results(g, tree, tau, l), want)
    both = together(g, (whole, tree), tau)
    same(*both)
    moved = [torch.flip(a, (0,)).contiguous() for a in l]
    for t in (whole, tree):
        ctx.refit_light_tree(t, *moved)
    same(results(g, tree, tau, moved), results(g, whole, tau, moved))
    tree.free()
    whole.free()
    assert used() == kept
print("ok")
"""


def test_hierarchies_without_paired_records(tmp_path_factory):
    assert fake_lib.run(fake_lib.build(tmp_path_factory), LIGHTS).strip().endswith("ok")
