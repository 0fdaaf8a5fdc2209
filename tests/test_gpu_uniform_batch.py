"""A batch whose frames all have one vertex form runs the batch frame compiled for
that form: every form, at the weight widths of the closing-in camera, instances
at different points of the path, with and without the point cache in the sphere
forms. States equal the oracle's and the exported vertices bit for bit."""
import numpy as np
import pytest

from oracle import Oracle
from tests.gpu_helpers import assert_same_state
from tests.test_gpu_forms import D, FORMS, _scene


@pytest.mark.gpu
@pytest.mark.parametrize("form", FORMS)
def test_one_form(form):
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    mesh, max_depth, frames = _scene(form)
    n = 3
    gs = [P.CBT(mesh, D - b, max_depth, point_cache=form.startswith("sphere") and b == 1) for b in range(n)]
    os_ = [Oracle(mesh, D - b, max_depth) for b in range(n)]
    batch = P.Batch(gs)
    rows = torch.zeros((n, 1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k in range(len(frames) - 2 * n):
        fps = [frames[k + 2 * b] for b in range(n)]
        batch.update(fps, vertices_out=list(rows))
        for b, (g, o, fp) in enumerate(zip(gs, os_, fps)):
            o.update(fp)
            assert g.stats()["error"] == 0
            if k % 6 == 5:
                assert_same_state(g, o, f"{form} frame {k} instance {b}")
                want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
                got = rows[b, :o.live_count].cpu().numpy()
                assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"{form} frame {k} instance {b}"
