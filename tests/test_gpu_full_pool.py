"""Pools filled to the brim and emptied again: forced splits until the gate
denies most of them, forced merges whose requests exceed the free slots (the
gate then looks for the tile in which they do), random requests in between. The
states and counts equal the oracle's frame by frame, in the single-instance,
the batch and the per-step frame, from pools of one word to several hundred
scan tiles."""
import pytest

import workloads as W
from oracle import Oracle
from tests.gpu_helpers import assert_same_state
from workloads.cameras import MODE_FORCE_MERGE, MODE_FORCE_SPLIT, MODE_RANDOM, forced_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gate", [0, 1], ids=["chain", "paper"])
@pytest.mark.parametrize("form", ["single", "batch", "per_step"])
@pytest.mark.parametrize("D", [5, 9, 13, 20])
def test_full_pool(D, form, gate):
    import paper_2407_02215_gb300 as P
    P.build_library()
    mesh = W.meshes.cube_mesh() if D >= 9 else W.meshes.tetra_mesh()
    depth = 22 if D == 20 else 12
    frames = [forced_params(MODE_FORCE_SPLIT, gate=gate) for _ in range(D + 2)]
    frames += [forced_params(MODE_FORCE_MERGE, gate=gate), forced_params(MODE_RANDOM, seed=D, gate=gate),
               forced_params(MODE_FORCE_SPLIT, gate=gate), forced_params(MODE_FORCE_MERGE, gate=gate),
               forced_params(MODE_FORCE_MERGE, gate=gate)]
    n = 2 if form == "batch" else 1
    gs, o = [P.CBT(mesh, D, depth) for _ in range(n)], Oracle(mesh, D, depth)
    batch = P.Batch(gs) if n > 1 else None
    gs[0].set_fused(form != "per_step")
    crossed = False
    for k, fp in enumerate(frames):
        if batch:
            batch.update([fp] * n)
        else:
            gs[0].update(fp)
        so = o.update(fp)
        crossed = crossed or so["merge_granted"] < so["merge_candidates"]
        for g in gs:
            sg = g.stats()
            assert sg["error"] == 0
            for key in ("live_after", "split_granted", "merge_granted", "allocated", "merge_candidates"):
                assert sg[key] == so[key], f"frame {k}: {key} gpu {sg[key]} oracle {so[key]}"
            if D < 20 or k % 4 == 3 or k >= len(frames) - 4:
                assert_same_state(g, o, f"frame {k}")
    assert crossed or gate == 1
