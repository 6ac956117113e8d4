"""Partitions of many segments: windows that the segment cuts shorter than the
triangle limit, segments scanned by warps and by blocks, at either side of that
line, the segments' batches counted by one block above 16,384 segments.  The starts must equal the
oracle's exactly; and the cost has to grow with the segments, not with their
square."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B

pytestmark = pytest.mark.gpu


def _starts(indices, max_unique, max_tris, segment, kept):
    import torch
    import paper_1805_08893_gb300 as gp
    idx = torch.from_numpy(indices.view(np.int32).copy()).cuda()
    starts = torch.full((indices.size // 3 + 1,), -7, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream()
    if kept:
        ctx = gp.gp_create("hash", mode=gp.GP_BATCH_DYNAMIC, max_unique=max_unique, max_tris=max_tris,
                           segment_tris=segment, stream=stream)
        part, n = gp.gp_partition(ctx, idx)
        gp.gp_partition_starts(ctx, part, starts)
        gp.gp_destroy(ctx)
    else:
        count = torch.zeros(1, dtype=torch.int32, device="cuda")
        gp.gp_partition_noalloc(idx, max_unique, max_tris, segment, starts, count, stream)
        torch.cuda.synchronize()
        n = int(count.item())
    return starts.cpu().numpy()[: n + 1].astype(np.int64)


MESHES = {"grid": lambda T: mg.grid_mesh(220).indices[: 3 * T], "random": lambda T: mg.random_indices(1, T, 9001)}


@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("tris,max_unique,max_tris,segment", [
    (72960, 16, 341, 32), (72928, 16, 341, 32),  # windows of 32: warps from 2,280 segments on, and one less
    (72960, 3, 1365, 32), (91200, 256, 1, 32),
    (90001, 256, 341, 63), (90001, 64, 64, 33), (40001, 20, 80, 20), (40001, 256, 341, 128), (40001, 256, 341, 129),
    (95000, 4096, 1365, 100), (95000, 3, 1, 40), (95000, 4096, 1365, 256), (95000, 768, 256, 256), (95000, 767, 256, 256),
    (16384, 256, 341, 1), (16385, 256, 341, 1), (33333, 4, 7, 2),  # either side of the count by one block
])
@pytest.mark.parametrize("kept", [False, True])
def test_many_segments(mesh, tris, max_unique, max_tris, segment, kept):
    indices = MESHES[mesh](tris).copy()
    indices[7] = 0xFFFFFFFF  # the reserved value is one id like any other here
    want = np.asarray(B.dynamic_partition(indices, max_unique, max_tris, segment), dtype=np.int64)
    assert np.array_equal(_starts(indices, max_unique, max_tris, segment, kept), want)


def test_cost_of_many_segments():
    # 2M segments of one triangle: ~2M blocks of ~4 us, some 5,000 at a time, are 2 ms.  When every eight of them
    # add up all the counts before them, 2M^2 / 16 counts are 1 TB to read, 100 ms at L2 rates
    import torch
    import paper_1805_08893_gb300 as gp
    T = 2_000_000
    idx = torch.arange(3 * T, dtype=torch.int32, device="cuda")
    ctx = gp.gp_create("hash", mode=gp.GP_BATCH_DYNAMIC, segment_tris=1, stream=torch.cuda.current_stream())
    try:
        def once():
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            part, n = gp.gp_partition(ctx, idx)
            b.record()
            torch.cuda.synchronize()
            gp.gp_partition_release(ctx, part)
            assert n == T
            return a.elapsed_time(b)

        once()
        assert min(once() for _ in range(3)) < 30
    finally:
        gp.gp_destroy(ctx)
