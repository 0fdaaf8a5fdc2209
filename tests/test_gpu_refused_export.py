"""cbt_vertices into a buffer that is too small for the live count: the call is
refused (CBT_ENOMEM) and reports the count, and nothing else changes: no row is
written, and coordinates outside the fixed-point range, which an accepted call
would note in the state's error word, are not looked at."""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from oracle import Oracle
from tests.gpu_helpers import assert_same_state

CBT_ENOMEM = 4


@pytest.mark.gpu
@pytest.mark.parametrize("short", [1, 100])
def test_refused_export_leaves_the_state(short):
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    spec = W.configs.config1(n_frames=6)
    g, o = P.CBT(spec.mesh, spec.D, spec.max_depth), Oracle(spec.mesh, spec.D, spec.max_depth)
    for fp in spec.frames[:4]:
        g.update(fp)
        o.update(fp)
    n = o.live_count
    rows = torch.full((n, 3, 3), 7.0, dtype=torch.float32, device="cuda")
    far, count = (C.c_double * 3)(1e9, -1e9, 1e9), C.c_uint32(0)  # 1e9 2^60 is far outside 62 bits
    rc = P.load().cbt_vertices(g.handle, C.c_void_p(rows.data_ptr()), far, 1, 60, n - short, C.byref(count), None)
    assert rc == CBT_ENOMEM and count.value == n
    torch.cuda.synchronize()
    assert bool((rows == 7.0).all())
    assert g.stats()["error"] == 0
    for fp in spec.frames[4:]:
        g.update(fp)
        o.update(fp)
        assert g.stats()["error"] == 0
        assert_same_state(g, o, "after the refused call")
    got = g.vertices((0.0, 0.0, 0.0)).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), o.vertices(np.zeros(3), 0, 20).view(np.uint32))
