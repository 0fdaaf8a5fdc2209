"""Every vertex form at every weight width: a camera that closes in on a point
of the surface until bisectors are refined to depths at which the exact weights
leave FP32 (24 bits), the fixed-point form's 48-bit products and FP64's 53
bits. The states equal the oracle's frame by frame and the exported vertices
bit for bit, in the one-launch and the per-step forms and in a batch whose
frames have different forms. Everything compared is exact; no tolerance."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle
from tests.gpu_helpers import assert_same_state
from workloads.cameras import PREC_FIXED, PREC_FP32, PREC_FP64, PREC_SPHERE

D = 13
FRAMES = 64
FORMS = {
    "fp32": dict(precision=PREC_FP32),
    "fp32_displaced": dict(precision=PREC_FP32, disp_amplitude=1e-4, disp_frequency=3.0, disp_octaves=4, disp_seed=5),
    "fixed_20": dict(precision=PREC_FIXED, fixed_shift=20),
    "fixed_40": dict(precision=PREC_FIXED, fixed_shift=40),
    "fixed_58": dict(precision=PREC_FIXED, fixed_shift=58),  # sums beyond 95 bits
    "fp64": dict(precision=PREC_FP64),
    "sphere": dict(precision=PREC_SPHERE, sphere_radius=1.0),
    "sphere_displaced": dict(precision=PREC_SPHERE, sphere_radius=1.0, disp_amplitude=1e-4, disp_frequency=3.0,
                             disp_octaves=3, disp_seed=7),
}


def _scene(form):
    """Mesh, maximum depth and the frames: straight down onto an interior
    point of a root triangle, the altitude halved every second frame."""
    kw = FORMS[form]
    sphere = kw["precision"] == PREC_SPHERE
    mesh = W.meshes.dodecahedron_mesh(1.0) if sphere else W.meshes.tetra_mesh()
    n = int(mesh.face_sizes[0])
    P = mesh.pos[mesh.face_verts[:n]]
    a, b, c = P[0], P[1], P.sum(0) / n
    target = 0.3 * a + 0.3 * b + 0.4 * c
    nrm = np.cross(b - a, c - a)
    nrm /= np.linalg.norm(nrm)
    if sphere:
        nrm = target / np.linalg.norm(target)
        target = nrm
    frames = []
    for k in range(FRAMES):
        eye = target + nrm * 2.0 ** (1 - k / 2)
        cam = W.cameras.Camera(eye=eye, target=target - nrm, up=b - a)
        frames.append(W.cameras.frame_params(cam, 180.0, **kw))
    return mesh, 50 if sphere else 56, frames


def _deepest(heap, H):
    return max(int(j).bit_length() for j in heap) - 1 - max(0, (H - 1).bit_length())


@pytest.mark.parametrize("form", FORMS)
def test_scene_reaches_the_widths(form):
    mesh, max_depth, frames = _scene(form)
    o = Oracle(mesh, D, max_depth)
    deepest = 0
    for fp in frames:
        assert o.update(fp)["ab_mismatch"] == 0
        deepest = max(deepest, _deepest(o.leaves()[1], mesh.H))
    assert deepest > (24 if form.startswith(("fp32", "fixed_20")) or "displaced" in form else 48), deepest


@pytest.mark.gpu
@pytest.mark.parametrize("fused", [True, False], ids=["fused", "per_step"])
@pytest.mark.parametrize("form", FORMS)
def test_deep_refinement(form, fused):
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    mesh, max_depth, frames = _scene(form)
    g, o = P.CBT(mesh, D, max_depth), Oracle(mesh, D, max_depth)
    g.set_fused(fused)
    rows = torch.zeros((1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k, fp in enumerate(frames):
        g.update(fp, vertices_out=rows)
        o.update(fp)
        assert g.stats()["error"] == 0
        assert_same_state(g, o, f"{form} frame {k}")
        want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
        got = rows[:o.live_count].cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"{form} frame {k}: vertices"


@pytest.mark.gpu
@pytest.mark.parametrize("fused", [True, False], ids=["fused", "per_step"])
def test_batch_of_all_forms(fused):
    """The instances' forms rotate every frame, so the batch runs as mixed
    forms throughout; with a single form in between."""
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    names = [n for n in FORMS if not n.startswith("sphere")]
    scenes = [_scene(n) for n in names]
    gs = [P.CBT(m, D, md) for m, md, _ in scenes]
    os_ = [Oracle(m, D, md) for m, md, _ in scenes]
    batch = P.Batch(gs)
    batch.set_fused(fused)
    rows = torch.zeros((len(gs), 1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k in range(0, 40):
        fps = [scenes[0 if k % 8 == 7 else (b + k) % len(names)][2][k] for b in range(len(gs))]
        batch.update(fps, vertices_out=list(rows))
        for b, (g, o, fp) in enumerate(zip(gs, os_, fps)):
            o.update(fp)
            if k % 5 == 4 or k % 8 == 7:
                assert g.stats()["error"] == 0
                assert_same_state(g, o, f"frame {k} instance {b}")
                want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
                got = rows[b, :o.live_count].cpu().numpy()
                assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"frame {k} instance {b}"


@pytest.mark.gpu
@pytest.mark.parametrize("sphere", [False, True], ids=["flat", "sphere"])
def test_form_changing_every_frame(sphere):
    """One instance of a small mesh whose frames change form, and now and then
    execution form: its root table is rewritten in another layout each time."""
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    names = [n for n in FORMS if n.startswith("sphere") == sphere]
    scenes = {n: _scene(n) for n in names}
    mesh, max_depth, _ = scenes[names[0]]
    g, o = P.CBT(mesh, D, max_depth, point_cache=sphere), Oracle(mesh, D, max_depth)
    rows = torch.zeros((1 << D, 3, 3), dtype=torch.float32, device="cuda")
    for k in range(40):
        fp = scenes[names[k % len(names)]][2][k // 2]
        g.set_fused(k % 11 != 7)
        g.update(fp, vertices_out=rows)
        o.update(fp)
        assert g.stats()["error"] == 0
        assert_same_state(g, o, f"frame {k}")
        want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
        got = rows[:o.live_count].cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"frame {k}: vertices"


@pytest.mark.gpu
def test_separate_triangles_displaced():
    """t triangles that share no point: a warp's 32 bisectors have from a few
    up to more than 64 distinct points, so its displaced points are evaluated
    in a part of a pass, one pass and two. Exact, as above."""
    import torch

    import paper_2407_02215_gb300 as P
    P.build_library()
    rng = np.random.default_rng(11)
    for t in (1, 2, 4, 5, 6, 8, 9, 10, 11, 12, 21, 22, 33):
        pos = rng.uniform(-1.0, 1.0, (t, 1, 3)) * [4.0, 4.0, 0.0] + rng.uniform(0.2, 1.0, (t, 3, 3)) * [[1, 0, 0], [0, 1, 0], [-1, -1, 0]]
        mesh = W.meshes._mesh("separate", np.arange(3 * t).reshape(t, 3).tolist(), pos)
        eye = np.array([0.1, 0.2, 3.0])
        fp = W.cameras.frame_params(W.cameras.Camera(eye=eye, target=eye - [0.0, 0.0, 1.0], up=[0.0, 1.0, 0.0]), 180.0,
                                    precision=PREC_FP32, disp_amplitude=0.05, disp_frequency=3.0, disp_octaves=6, disp_seed=5)
        g, o = P.CBT(mesh, 10, 12), Oracle(mesh, 10, 12)
        rows = torch.zeros((1 << 10, 3, 3), dtype=torch.float32, device="cuda")
        for k in range(4):
            g.update(fp, vertices_out=rows)
            o.update(fp)
            assert g.stats()["error"] == 0
            assert_same_state(g, o, f"{t} triangles frame {k}")
            want = o.vertices(fp.eye, fp.precision, fp.fixed_shift, fp.sphere_radius, frame=fp)
            got = rows[:o.live_count].cpu().numpy()
            assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), f"{t} triangles frame {k}: vertices"
