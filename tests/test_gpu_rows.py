"""Static batches with rows for a third of their indices: batches that hold
fewer unique vertices than that, about as many, and all of them distinct, over
every dedup method, shader and block size that takes the smaller
configuration.  Outputs must equal the naive kernel's bit for bit (the same
shader code) and the counts the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu


def _meshes():
    grid = mg.grid_mesh(64)
    V = 6000
    rng = np.random.default_rng(11)
    distinct = np.concatenate([rng.permutation(V)[:V - V % 3] for _ in range(4)]).astype(np.uint32)  # no repeats near
    some = (rng.integers(0, 300, size=9000) + 5 * (np.arange(9000) // 768)).astype(np.uint32)  # ~250 of 768 unique
    return {"grid": grid, "distinct": mg.Mesh(mg.random_vertices(1, V), distinct, mg.FMT_PNU32, "distinct"),
            "some": mg.Mesh(mg.random_vertices(2, V), some, mg.FMT_PNU32, "some")}


MESHES = _meshes()


@pytest.mark.parametrize("which", list(MESHES))
@pytest.mark.parametrize("variant,S_,threads", [("hash", 768, 256), ("phash", 768, 256), ("sort", 768, 256),
                                                ("hash", 192, 128), ("hash", 381, 64), ("phash", 1023, 512),
                                                ("hash", 1023, 256)])
@pytest.mark.parametrize("shader", ["mvp", "skin", "envelope"])
def test_rows_for_a_third(which, variant, S_, threads, shader):
    mesh, palette = MESHES[which], None
    if shader == "skin":
        mesh, palette = mg.skin_mesh(mesh, 3)
    sid = {"mvp": S.SHADER_MVP, "skin": S.SHADER_SKIN, "envelope": S.SHADER_ENVELOPE}[shader]
    uni, _ = uniforms_for(mesh, sid, palette=palette)
    want = draw_gpu(mesh, "naive", sid, "static", uni)
    got = draw_gpu(mesh, variant, sid, "static", uni, batch_indices=S_, threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.ids, mesh.indices)
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
    assert np.array_equal(got.inv, B.unique_per_batch(mesh.indices, B.static_starts(mesh.num_tris, S_)))


def test_captured_draws_replayed_side_by_side():
    """Two draws of one context, each captured into a graph, replayed on two streams at once: neither may use memory
    of the other's (every batch holds more unique vertices than a third of its indices)."""
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = MESHES["distinct"]
    rng = np.random.default_rng(5)
    big = mg.Mesh(mesh.vertices, np.concatenate([rng.permutation(6000) for _ in range(200)]).astype(np.uint32), mesh.fmt,
                  "big")
    uni, _ = uniforms_for(big, S.SHADER_MVP)
    want = draw_gpu(big, "naive", S.SHADER_MVP, "static", uni, debug=False).out
    verts = torch.from_numpy(big.vertices).cuda()
    # the second graph draws the triangles in reverse order
    idx = [torch.from_numpy(i.view(np.int32).copy()).cuda()
           for i in (big.indices, np.ascontiguousarray(big.indices.reshape(-1, 3)[::-1]).reshape(-1))]
    out = [torch.zeros(big.num_tris * 21, device="cuda") for _ in idx]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctx = gp.gp_create("hash", stream=streams[0], batch_indices=768)
    try:
        graphs = []
        for i, o in zip(idx, out):
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=streams[0]):
                gp.gp_submit_drawcall(ctx, i, verts, gp.GP_SHADER_MVP, uni, o)
            graphs.append(graph)
        for _ in range(3):
            for o in out:
                o.zero_()
            torch.cuda.synchronize()
            for graph, stream in zip(graphs, streams):
                with torch.cuda.stream(stream):
                    graph.replay()
            torch.cuda.synchronize()
            want = want.reshape(big.num_tris, -1)
            for o, w in zip(out, (want, want[::-1])):
                assert np.array_equal(o.cpu().numpy().reshape(want.shape).view(np.uint32),
                                      np.ascontiguousarray(w).view(np.uint32))
        del graphs
    finally:
        gp.gp_destroy(ctx)
