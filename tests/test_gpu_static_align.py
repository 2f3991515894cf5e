"""The build without allocation writes into arrays the caller owns, at any address a caller may
have: a record array at an odd multiple of 16 bytes (the documented alignment), and of 4 and 8.
Equal, byte for byte, to the allocating build's hierarchy; the words around the array stay."""
import ctypes

import numpy as np
import pytest

from gpu_util import dev, upload_scene
from test_gpu_build import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 33, 512, 513, 3001])
@pytest.mark.parametrize("offset", [16, 48, 8, 4])
def test_records_at_any_word(ctx, n, offset):  # noqa: F811
    import torch
    import paper_1907_12343_gb300 as hrr
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3)).astype(np.float32)
    g = upload_scene({"light_pos": pos, "intensity": np.exp(rng.standard_normal(n)).astype(np.float32),
                      "eye_pos": pos[:1], "px": np.zeros(1, np.uint16), "py": np.zeros(1, np.uint16)})
    tree = ctx.build_light_tree(g["lx"], g["ly"], g["lz"], g["li"])
    nodes, perm = tree.download()
    n_rec, at = max(n - 1, 1), offset // 4
    buf = torch.full((16 * n_rec + 32,), 0x5A5A5A5A, dtype=torch.int32, device=dev())
    dev_perm = torch.full((n + 8,), -1, dtype=torch.int32, device=dev())
    assert buf.data_ptr() % 64 == 0
    height = ctypes.c_uint32(12345)
    err = ctypes.create_string_buffer(256)
    L = hrr.hrr_lights(*(g[k].data_ptr() for k in ("lx", "ly", "lz", "li")))
    st = hrr.hrr_build_light_tree_static(L, n, buf.data_ptr() + offset, dev_perm.data_ptr() + 4, ctypes.byref(height),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), err, 256)
    assert st == hrr.HRR_OK, err.value
    got = buf.cpu().numpy()
    if n > 1:  # a single light's record is not downloaded
        assert got[at:at + 16 * n_rec].tobytes() == nodes.tobytes()
    else:
        want = np.float32([*pos[0], g["li"].item()])
        assert np.array_equal(got[at:at + 4].view(np.float32), want) and np.array_equal(got[at + 8:at + 12].view(np.float32), want)
    assert (got[:at] == 0x5A5A5A5A).all() and (got[at + 16 * n_rec:] == 0x5A5A5A5A).all()
    p = dev_perm.cpu().numpy()
    assert np.array_equal(p[1:n + 1], perm.view(np.int32)) and p[0] == -1 and (p[n + 1:] == -1).all()
    assert height.value == tree.height
    tree.free()
