"""A batch in graph mode whose frames change form: each form's frames replay the
graph captured for it, so that a change costs a replay and no new capture. The
states equal the oracle's (exact), the launch count is that of the execution form
of the last frame, and a call on frames that alternate takes no longer on the host
than twice a call on frames that do not, plus 20 us (captured anew each time, a
per-step frame of this batch took 58.6 us, replayed 8.0)."""
import statistics
import time

import pytest

from oracle import Oracle
from tests.gpu_helpers import assert_same_state
from tests.test_gpu_forms import D, _scene

NAMES = ["fp32", "fp32_displaced", "fixed_40", "fp64"]


@pytest.fixture(scope="module")
def P():
    import paper_2407_02215_gb300 as P
    P.build_library()
    return P


@pytest.mark.gpu
def test_results_and_launch_counts(P):
    scenes = [_scene(n) for n in NAMES]
    mesh, max_depth, _ = scenes[0]
    gs, os_ = [P.CBT(mesh, D, max_depth) for _ in range(2)], [Oracle(mesh, D, max_depth) for _ in range(2)]
    batch = P.Batch(gs)
    batch.set_graph(True)
    for k in range(48):
        fused = (k // 5) % 2 == 0
        batch.set_fused(fused)
        # one form per frame; every third frame the instances differ
        fps = [scenes[(k + (b if k % 3 == 0 else 0)) % len(NAMES)][2][k] for b in range(2)]
        batch.update(fps)
        assert batch.last_launch_count == (1 if fused else 10)
        for b, (g, o, fp) in enumerate(zip(gs, os_, fps)):
            o.update(fp)
            assert g.stats()["error"] == 0
            assert_same_state(g, o, f"frame {k} instance {b}")


@pytest.mark.gpu
@pytest.mark.parametrize("fused", [True, False], ids=["fused", "per_step"])
def test_a_change_of_form_replays(P, fused):
    import torch
    scenes = [_scene(n) for n in NAMES[:2]]
    mesh, max_depth, _ = scenes[0]
    batch = P.Batch([P.CBT(mesh, D, max_depth) for _ in range(2)])
    batch.set_fused(fused)
    batch.set_graph(True)
    packed = [P.cbt.pack_frames([s[2][8]] * 2, "cuda") for s in scenes]

    def call_us(order):
        got = []
        for k in range(60):
            torch.cuda.synchronize()
            t = time.perf_counter()
            batch.update_packed(packed[order[k % len(order)]][0])
            got.append((time.perf_counter() - t) * 1e6)
        return statistics.median(got[10:])

    steady = max(call_us([0]), call_us([1]))
    alternating = call_us([0, 1])
    assert alternating <= 2.0 * steady + 20.0, f"{alternating:.1f} us alternating, {steady:.1f} us steady"
