"""Loop subdivision where its reads and writes have edges: rings read 16 bytes
at a time (rings of every length and offset, an array that is not 16-byte
aligned, the last ring at the array's end), and a warp's triangles written 16
at a time (batches that end inside a warp or a half of one).  Output within the
oracle's tolerance of positions of order 1: a ring's sum of at most 40 float32
terms, weighted by about one over their number, errs by at most 40 x 6e-8."""
import numpy as np
import pytest

import meshgen as mg
from oracle import loop as L

pytestmark = pytest.mark.gpu


def _fans(sizes, seed):
    """Closed fans of the given sizes side by side: inner vertices of that valence, outer ones on the boundary."""
    rng = np.random.default_rng(seed)
    pos, tris = [], []
    for k, n in enumerate(sizes):
        base = len(pos)
        pos.append([k / len(sizes), 0.0, 0.1])
        pos += [[k / len(sizes) + 0.01 * np.cos(t), 0.01 * np.sin(t), 0.0] for t in 2 * np.pi * np.arange(n) / n]
        tris += [[base, base + 1 + i, base + 1 + (i + 1) % n] for i in range(n)]
    verts = np.zeros((len(pos), 8), dtype=np.float32)
    verts[:, :3] = np.asarray(pos) + 0.001 * rng.standard_normal((len(pos), 3))
    return verts, np.asarray(tris, dtype=np.uint32).reshape(-1)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("variant,S", [("naive", 0), ("warp", 96), ("hash", 255), ("sort", 141), ("phash", 51)])
def test_rings_and_ragged_warps(shift, variant, S):
    import torch
    import paper_1805_08893_gb300 as gp
    verts, indices = _fans([3, 4, 5, 6, 7, 8, 9, 12, 13, 40, 6, 3], shift)
    off, ring, opp, flags = (torch.from_numpy(x.view(np.int32).copy()).cuda()
                             for x in gp.gp_loop_adjacency(indices, verts.shape[0]))
    at = torch.full((ring.numel() + shift,), -1, dtype=torch.int32, device="cuda")  # from entry 'shift' of it
    at[shift:] = ring
    idx = torch.from_numpy(indices.view(np.int32).copy()).cuda()
    T = indices.size // 3
    out = torch.full((T * 36 + 36,), float("nan"), device="cuda")
    cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
    gp.gp_loop_subdivide(idx, torch.from_numpy(verts).cuda(), (off, at[shift:], opp, flags), out, cnt, variant,
                         batch_indices=S, threads=64 if S else 0)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.isnan(got[36 * T:]).all()  # nothing past the end
    want = L.subdivide(verts[:, :3], indices)
    assert np.allclose(got[:36 * T].reshape(-1, 4, 3, 3), want, rtol=1e-5, atol=1e-5)
    assert int(cnt[2]) == 0
