"""A pool above the single-instance frame's tables (2^23 slots) whose live count
grows past the sizes at which its frame changes how it deals out the work.
Classify and the walks take item tiles in parts while few bisectors live (at 608
blocks FP32 classify up to 304 tiles of 1,024, the other forms' up to 1,215, the
walks up to 152); tiles and parts are handed out by a counter once there are more
of them than blocks; the last part and the last tile are ragged. States and
counts equal the oracle's, the exported vertices bit for bit."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle
from tests.gpu_helpers import assert_same_state
from workloads.cameras import MODE_FORCE_MERGE, MODE_FORCE_SPLIT, MODE_RANDOM, PREC_FP32, forced_params

pytestmark = pytest.mark.gpu
D = 23


def _check(g, o, fp, rows, where, state):
    so, sg = o.update(fp), g.stats()
    assert sg["error"] == 0, where
    for key in ("live_after", "split_granted", "merge_granted", "split_bisectors", "merged_bisectors", "allocated",
                "merge_candidates"):
        assert sg[key] == so[key], f"{where}: {key} gpu {sg[key]} oracle {so[key]}"
    if state:
        assert_same_state(g, o, where)
        want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
        got = rows[:o.live_count].cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"{where}: vertices"


@pytest.fixture(scope="module")
def P():
    import paper_2407_02215_gb300 as P
    P.build_library()
    return P


@pytest.mark.parametrize("form", ["fp32", "displaced"])
def test_growing_and_shrinking(P, form):
    """From 24 bisectors by forced splits to 1.57 million, with a random frame
    at every second size and at the end merges."""
    import torch
    kw = {} if form == "fp32" else dict(precision=PREC_FP32, disp_amplitude=0.05, disp_frequency=3.0, disp_octaves=2,
                                        disp_seed=5)
    mesh = W.meshes.cube_mesh()
    g, o = P.CBT(mesh, D, 20), Oracle(mesh, D, 20)
    rows = torch.zeros((1 << D, 3, 3), dtype=torch.float32, device="cuda")
    modes = []
    for k in range(16):
        modes += [MODE_FORCE_SPLIT] + ([MODE_RANDOM] if k % 2 else [])
    modes += [MODE_FORCE_MERGE, MODE_RANDOM, MODE_FORCE_MERGE, MODE_FORCE_MERGE]
    for k, mode in enumerate(modes):
        fp = forced_params(mode, seed=k, **kw)
        g.update(fp, vertices_out=rows)
        _check(g, o, fp, rows, f"{form} frame {k}", k % 5 == 4 or k == len(modes) - 1)


@pytest.mark.parametrize("scene", ["grid", "terrain", "planet_fixed", "planet_fp64", "dodeca", "waves"])
def test_lod_frames(P, scene):
    """Camera frames of every vertex form, a few thousand to some 100,000 bisectors."""
    import torch
    C = W.configs
    spec = {"grid": lambda: C.config2(n_frames=12, tau_px=4.0, nx=24),
            "terrain": lambda: C.config_terrain(n_frames=12, nx=24, D=20),
            "planet_fixed": lambda: C.config3(n_frames=600, tau_px=12.0),
            "planet_fp64": lambda: C.config3(n_frames=600, tau_px=12.0, precision=W.cameras.PREC_FP64),
            "dodeca": lambda: C.config_dodeca(), "waves": lambda: C.config_waves()}[scene]()
    frames = spec.frames if len(spec.frames) <= 12 else spec.frames[100:520:35]
    g, o = P.CBT(spec.mesh, D, spec.max_depth), Oracle(spec.mesh, D, spec.max_depth)
    rows = torch.zeros((1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k, fp in enumerate(frames):
        g.update(fp, vertices_out=rows)
        _check(g, o, fp, rows, f"{scene} frame {k}", k % 4 == 3 or k == len(frames) - 1)
