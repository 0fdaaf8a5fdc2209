"""The single-instance frame's export of more rows than a block's list of
uncached rows holds: forced splits, in which no vertex is cached by a LOD test,
until 1.57 million bisectors are live (2,600 rows per block of a full grid; the
list is evaluated when it passes 1,536). The displaced and the projected form;
every row equals the oracle's bit for bit."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle
from workloads.cameras import MODE_FORCE_SPLIT, PREC_FP32, PREC_SPHERE, forced_params

FORMS = {
    "displaced": dict(precision=PREC_FP32, disp_amplitude=0.05, disp_frequency=3.0, disp_octaves=2, disp_seed=5),
    "sphere": dict(precision=PREC_SPHERE, sphere_radius=1.0),
}


@pytest.mark.gpu
@pytest.mark.parametrize("form", FORMS)
def test_list_passes_its_limit(form):
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    D = 22
    mesh = W.meshes.cube_mesh()
    fp = forced_params(MODE_FORCE_SPLIT, **FORMS[form])
    g, o = P.CBT(mesh, D, 16), Oracle(mesh, D, 16)
    rows = torch.zeros((1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k in range(16):
        g.update(fp, vertices_out=rows if k >= 14 else None)
        o.update(fp)
        if k >= 14:
            assert g.stats()["error"] == 0
            assert g.live_count() == o.live_count == 24 << (k + 1)
            want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
            got = rows[:o.live_count].cpu().numpy()
            assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"frame {k}"
