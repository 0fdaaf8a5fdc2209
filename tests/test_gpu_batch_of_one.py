"""A batch of one instance and cbt_update taking turns on the same state. Both
run the single-instance frame, which leaves what the next frame starts from (the
free list, the ones before each word tile, cleared counters) with the instance:
whichever handle launches the next frame has to find it. The batches' own memory
holds garbage at first. States, counts and vertices equal the oracle's frame by
frame; everything compared is exact."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle
from tests.gpu_helpers import assert_same_state
from workloads.cameras import MODE_FORCE_MERGE, MODE_FORCE_SPLIT, MODE_RANDOM, forced_params

pytestmark = pytest.mark.gpu

# who launches each frame: u cbt_update, a and b two batches of one, s cbt_update per step
TURNS = ["uau", "uabuab", "ab", "uaas", "uuab", "su"]


def _scene(scene):
    if scene == "cube":  # at most 64 halfedges: the frame without a barrier after its first phase
        spec = W.configs.config1(n_frames=24)
        return spec.mesh, 14, spec.max_depth, spec.frames
    if scene == "grid":
        spec = W.configs.config2(n_frames=24, nx=24)
        return spec.mesh, 16, spec.max_depth, spec.frames
    frames = [forced_params(MODE_FORCE_SPLIT) for _ in range(13)]  # the pool runs full
    frames += [forced_params(MODE_RANDOM, seed=3), forced_params(MODE_FORCE_MERGE)] * 3
    return W.meshes.cube_mesh(), 13, 12, frames


@pytest.mark.parametrize("turns", TURNS)
@pytest.mark.parametrize("scene", ["cube", "grid", "full"])
def test_turns_on_one_state(scene, turns):
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    lib = P.load()
    mesh, D, max_depth, frames = _scene(scene)
    g, o = P.CBT(mesh, D, max_depth), Oracle(mesh, D, max_depth)
    batches = {}
    for name in "ab":
        nbytes = lib.cbt_batch_workspace_bytes(P.cbt.handles_of([g]), 1)
        garbage = torch.full((nbytes,), 0xA5, dtype=torch.uint8, device="cuda")
        del garbage  # the batch's memory comes from the same block
        batches[name] = P.Batch([g])
    rows = torch.zeros((1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k, fp in enumerate(frames):
        who = turns[k % len(turns)]
        g.set_fused(who != "s")
        if who in batches:
            batches[who].update([fp], vertices_out=[rows])
        else:
            g.update(fp, vertices_out=rows)
        so, sg = o.update(fp), g.stats()
        where = f"frame {k} by {who}"
        assert sg["error"] == 0, where
        for key in ("live_after", "split_granted", "merge_granted", "allocated", "merge_candidates"):
            assert sg[key] == so[key], f"{where}: {key} gpu {sg[key]} oracle {so[key]}"
        assert_same_state(g, o, where)
        want = o.vertices(fp.eye, fp.precision, fp.fixed_shift)
        got = rows[:o.live_count].cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"{where}: vertices"
