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


SCENES = HEAD + """
rng = np.random.default_rng(4)
n_s = 20000
x = [torch.from_numpy(a.astype(np.float32)).to(dev()) for a in rng.random((6, n_s))] + [torch.ones(n_s, device=dev())]
pairs = torch.arange(n_s, dtype=torch.int32, device=dev()).repeat_interleave(2).view(n_s, 2).contiguous()
sums = torch.zeros(n_s, device=dev())

def visible(scene):
    v = torch.zeros(n_s, dtype=torch.uint8, device=dev())
    ctx.connect(*x[:3], tuple(x[3:]), 1e-3, pairs, n_s, scene=scene, visible=v, eye_sum=sums)
    return v.cpu().numpy()

for n, spread in ((2, 1.0), (300, 1.0), (150000, 1.0), (150000, 1e-9)):
    tris = 0.5 + spread * (rng.random((n, 1, 3)) - 0.5) + 0.5 * n ** -0.5 * rng.standard_normal((n, 3, 3))
    if spread < 1:  # the keys of one cell: a full sort
        tris += 0.5 - tris.mean(axis=1, keepdims=True)
    t = torch.from_numpy(tris.reshape(n, 9).astype(np.float32)).to(dev())
    scene = ctx.build_scene(t)
    want, kept = visible(scene), used()
    assert 0 < want.sum() < n_s or n == 2
    os.environ["HRR_FAKE_MEMORY"] = str(kept + 257 * n + (1 << 16))
    tight = ctx.build_scene(t)
    assert np.array_equal(visible(tight), want)
    os.environ["HRR_FAKE_MEMORY"] = str(kept + 192 * (n - 1))
    try:
        ctx.build_scene(t)
        raise SystemExit("built without memory")
    except hrr.HRRError as e:
        assert e.status == hrr.HRR_ERR_OOM, e
    del os.environ["HRR_FAKE_MEMORY"]
    tight.free()
    scene.free()
    assert used() == 0
print("ok")
"""


def test_scenes_build_in_the_memory_of_their_nodes(tmp_path_factory):
    assert fake_lib.run(fake_lib.build(tmp_path_factory), SCENES).strip().endswith("ok")
