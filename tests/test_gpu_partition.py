"""GPU parity of the dynamic partition's scan (Section 3.4) at the edges of
its launch shapes: one, two or four indices per thread, windows cut by the
unique limit or the triangle limit, segments of odd lengths, ragged ends.
The batch starts must equal the oracle's greedy scan exactly."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B

pytestmark = pytest.mark.gpu


def _starts(indices, max_unique, max_tris, segment):
    import torch
    import paper_1805_08893_gb300 as gp
    idx = torch.from_numpy(indices.view(np.int32).copy()).cuda()
    starts = torch.full((indices.size // 3 + 1,), -7, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    gp.gp_partition_noalloc(idx, max_unique, max_tris, segment, starts, count, torch.cuda.current_stream())
    torch.cuda.synchronize()
    return starts.cpu().numpy()[: int(count.item()) + 1].astype(np.int64)


# locality (windows taken whole), none (windows cut), and a change from one to the other within a segment
MESHES = {"grid": lambda: mg.grid_mesh(64).indices,
          "random": lambda: mg.random_indices(1, 5003, 4000),
          "mixed": lambda: np.concatenate([mg.grid_mesh(40).indices, mg.random_indices(2, 1500, 1600),
                                           mg.grid_mesh(33).indices])}


@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("max_unique,max_tris", [(3, 1), (4, 2), (5, 11), (64, 64), (90, 128), (100, 129), (256, 256),
                                                 (200, 257), (256, 341), (320, 426), (4096, 683), (700, 1365),
                                                 (4096, 1365)])
def test_window_edges(mesh, max_unique, max_tris):
    indices = MESHES[mesh]()
    want = np.asarray(B.dynamic_partition(indices, max_unique, max_tris, 4096), dtype=np.int64)
    assert np.array_equal(_starts(indices, max_unique, max_tris, 4096), want)


@pytest.mark.parametrize("tris", [1, 2, 5, 63, 64, 65, 341, 342, 4095, 4096, 4097, 4999])
@pytest.mark.parametrize("segment", [1, 7, 1000, 0xFFFFFFFF])
def test_segments_and_ragged_ends(tris, segment):
    indices = MESHES["mixed"]()[: 3 * tris]
    if tris > 3:
        indices = indices.copy()
        indices[4] = 0xFFFFFFFF  # the reserved value is one id like any other here
    want = np.asarray(B.dynamic_partition(indices, 256, 341, 0 if segment == 0xFFFFFFFF else segment),
                      dtype=np.int64)
    assert np.array_equal(_starts(indices, 256, 341, segment), want)
