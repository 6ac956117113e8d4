"""Loop subdivision at both sides of the line between its batched kernels: blocks of
twice as many threads as a batch has triangles, and of fewer; blocks whose last
warps have no triangle to write.  Every method writes the same bits as the naive
one, and nothing past the end."""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

MESHES = {"sphere": mg.geodesic_sphere(14, 2), "grid": mg.grid_mesh(40)}


def _draw(mesh, variant, torch, gp, **more):
    idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
    verts = torch.from_numpy(mesh.vertices).cuda()
    adj = [torch.from_numpy(x.view(np.int32).copy()).cuda()
           for x in gp.gp_loop_adjacency(mesh.indices, mesh.vertices.shape[0])]
    out = torch.full((mesh.num_tris * 36 + 64,), float("nan"), device="cuda")
    cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
    gp.gp_loop_subdivide(idx, verts, adj, out, cnt, variant, **more)
    torch.cuda.synchronize()
    assert int(cnt[2]) == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("which", list(MESHES))
@pytest.mark.parametrize("variant", ["hash", "phash", "sort"])
@pytest.mark.parametrize("S,threads", [(3, 32), (48, 32), (51, 32), (96, 64), (99, 64), (96, 128), (96, 256), (192, 128),
                                       (195, 128), (768, 512), (771, 512), (768, 256), (1536, 64), (4095, 512)])
def test_same_bits(which, variant, S, threads):
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = MESHES[which]
    want = _draw(mesh, "naive", torch, gp)
    got = _draw(mesh, variant, torch, gp, batch_indices=S, threads=threads)
    assert np.isnan(got[36 * mesh.num_tris:]).all()
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
