"""How many batch tallies a run takes (CPU): never more than a launch can use,
and no more memory than leaves room for other handles and programs."""
import pytest

GiB = 1 << 30
ALL = (280 * GiB, 284 * GiB, 0)
BODY = 512 * 512 * 600           # 1.26 GB a tally


@pytest.fixture(scope="module")
def slots():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    return nmdose.load().nm_debug_batch_slots


@pytest.mark.parametrize("voxels,n,batches,memory,want", [
    (64**3, 10**6, 10, ALL, 10), (64**3, 10**6, 16, ALL, 16), (64**3, 10**6, 33, ALL, 11), (64**3, 10**6, 1, ALL, 1),
    # batches that share no launch: below 64 histories, or above 2^31 a launch
    (64**3, 639, 10, ALL, 1), (64**3, 640, 10, ALL, 10), (64**3, 10 << 31, 10, ALL, 1), (64**3, 10 << 30, 10, ALL, 2),
    (64**3, 10 * ((1 << 31) // 3), 10, ALL, 3), (64**3, (10 << 31) // 3, 10, ALL, 2),   # three of the larger: one above
    # 16 GiB a handle, slot x voxel below 2^32
    (BODY, 10**9, 10, ALL, 10), (2**31 - 1, 10**9, 10, (2**60, 2**60, 0), 1), (2**28, 10**9, 10, (2**60, 2**60, 0), 5),
    # a quarter of what is free, beyond the first
    (BODY, 10**9, 10, (20 * GiB, 284 * GiB, 0), 5), (BODY, 10**9, 10, (4 * GiB, 284 * GiB, 0), 1),
    (BODY, 10**9, 10, (0, 284 * GiB, 0), 1),
    # an eighth of the device for all handles
    (BODY, 10**9, 10, (200 * GiB, 284 * GiB, 30 * GiB), 5), (BODY, 10**9, 10, (200 * GiB, 284 * GiB, 40 * GiB), 1)])
def test_batch_slots(slots, voxels, n, batches, memory, want):
    assert slots(voxels, n, batches, *memory) == want


def test_many_handles_leave_room(slots):
    """Thirty whole-body handles, 6 GiB each by themselves, fit a device as they did with one tally each."""
    free, total, held = 280 * GiB, 284 * GiB, 0
    for _ in range(30):
        free -= 6 * GiB
        extra = (slots(BODY, 10**9, 10, free, total, held) - 1) * 8 * BODY
        free, held = free - extra, held + extra
        assert free > 0 and held <= total // 8
