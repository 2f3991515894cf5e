"""A wait of the sort that runs out (its first tile is never taken, so nothing publishes the counts
the others wait for): every build reports HRR_ERR_TIMEOUT, and the context and the device go on as
before."""
import pytest

import fake_lib

pytestmark = pytest.mark.gpu

SCRIPT = """
import ctypes, os
import numpy as np, torch
import paper_1907_12343_gb300 as hrr
assert hrr.__file__.startswith(os.getcwd())
dev = torch.device("cuda:0")
ctx = hrr.Context(0)
rng = np.random.default_rng(3)
n, small = 150000, 60000  # sizes at which the sort's scratch has room for a ticket more
pos = rng.random((n, 3)).astype(np.float32)
x = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (*pos.T, np.ones(n, np.float32))]
tris = torch.from_numpy(rng.random((n, 9)).astype(np.float32)).to(dev)

def light(topology):
    return lambda: ctx.build_light_tree(*x, topology=topology).download()

def scene():
    ctx.build_scene(tris).free()

def static():
    nodes = torch.zeros((small - 1, 16), dtype=torch.int32, device=dev)
    perm = torch.zeros(small, dtype=torch.int32, device=dev)
    err = ctypes.create_string_buffer(256)
    st = hrr.hrr_build_light_tree_static(hrr.hrr_lights(*(a.data_ptr() for a in x)), small, nodes.data_ptr(),
                                         perm.data_ptr(), None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream),
                                         err, 256)
    if st:
        raise hrr.HRRError(st, err.value.decode())
    return nodes.cpu().numpy(), perm.cpu().numpy()

calls = [light("radix"), light("cost"), scene, static]
before = [f() for f in calls]
os.environ["HRR_FAKE_TICKETS"] = "1"
for f in calls:
    try:
        f()
        raise SystemExit("the wait did not run out")
    except hrr.HRRError as e:
        assert e.status == hrr.HRR_ERR_TIMEOUT, e
del os.environ["HRR_FAKE_TICKETS"]
torch.cuda.synchronize()
after = [f() for f in calls]
for a, b in zip(before, after):
    if a is not None:
        assert all(p.tobytes() == q.tobytes() for p, q in zip(a, b))
print("ok")
"""


def test_a_wait_that_runs_out_is_a_timeout(tmp_path_factory):
    assert fake_lib.run(fake_lib.build(tmp_path_factory), SCRIPT).strip().endswith("ok")
