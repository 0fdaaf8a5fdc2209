"""What an instance's workspace costs per slot (host only): 116 bytes in the slot
arrays, 12 in 32 slots' bitfield word and tree nodes, the batch's descriptors; the
single-instance frame's second free list and clear masks (4 bytes a slot and 4 a
word) only in pools that this frame takes, which end at 2^22 slots."""
import pytest


@pytest.mark.parametrize("D", range(16, 30))
def test_bytes_per_slot(D):
    import paper_2407_02215_gb300 as P
    P.build_library()
    assert P.workspace_bytes(24, D) % 256 == 0
    if D == 22:  # the next pool is without those arrays
        return
    grown = (P.workspace_bytes(24, D + 1) - P.workspace_bytes(24, D)) / 2.0 ** D
    most = 116 + 12 / 32 + 0.1 + (4 + 4 / 32 if D < 22 else 0)
    assert 116 <= grown <= most, grown


def test_largest_single_instance_pool():
    import paper_2407_02215_gb300 as P
    P.build_library()
    per_slot = [P.workspace_bytes(24, D) / 2.0 ** D for D in (22, 23)]
    assert 4.0 <= per_slot[0] - per_slot[1] <= 4.3, per_slot
