"""Captured draws and the context's other draws: a graph goes on writing the
record of its draw at every replay, so no other draw may use that record, and
folding tickets may not touch it.  The reuse kernel claims its last batches from
the record: a wrong one leaves triangles undrawn and shows in the counts."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,replays,captured", [("hash", 1, 1), ("phash", 2, 1), ("sort", 1, 1), ("naive", 1, 1),
                                                      ("hash", 1, 70)])
def test_plain_draws_after_replays(variant, replays, captured):
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = mg.grid_mesh(64)
    uni, _ = uniforms_for(mesh, S.SHADER_MVP)
    # 1,985 batches, more than blocks are resident: the last ones are claimed from the record
    cfg = {} if variant == "naive" else {"batch_indices": 12}
    want = torch.from_numpy(draw_gpu(mesh, "naive", S.SHADER_MVP, "static", uni, debug=False).out.reshape(-1)).cuda()
    idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
    verts = torch.from_numpy(mesh.vertices).cuda()
    out, out2 = torch.zeros_like(want), torch.zeros_like(want)
    inv = 3 * mesh.num_tris
    if variant != "naive":
        inv = int(B.batch_invocations(mesh.indices, B.static_starts(mesh.num_tris, 12), variant).sum())
    stream = torch.cuda.Stream()
    ctx = gp.gp_create(variant, stream=stream, **cfg)
    try:
        def draw(o):
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, o)

        with torch.cuda.stream(stream):
            draw(out)
        gp.gp_sync(ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(captured):
                draw(out2)
        with torch.cuda.stream(stream):
            draw(out)
        gp.gp_stats(ctx, reset=True)  # folds the captured tickets too
        equal = torch.ones((), dtype=torch.bool, device="cuda")
        torch.cuda.synchronize()
        plain = 1100  # once round the ring of records
        with torch.cuda.stream(stream):
            for k in range(plain):
                if k < replays or k % 100 == 50:
                    out2.fill_(float("nan"))
                    graph.replay()
                    equal &= torch.all(out2 == want)
                out.fill_(float("nan"))
                draw(out)
                equal &= torch.all(out == want)
                if k == 600:
                    gp.gp_sync(ctx)
        st = gp.gp_stats(ctx)
        assert bool(equal)
        assert st["draws"] == plain and st["invocations"] == plain * inv
        del graph
    finally:
        gp.gp_destroy(ctx)


def test_counts_of_a_replayed_draw():
    """A captured draw counts once, with what its last replay counted."""
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = mg.grid_mesh(64)
    uni, _ = uniforms_for(mesh, S.SHADER_MVP)
    idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
    verts = torch.from_numpy(mesh.vertices).cuda()
    out = torch.zeros(mesh.num_tris * 21, device="cuda")
    stream = torch.cuda.Stream()
    ctx = gp.gp_create("hash", stream=stream, batch_indices=12)
    try:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
        with torch.cuda.stream(stream):
            for _ in range(3):
                graph.replay()
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
        st = gp.gp_stats(ctx)
        inv = int(B.batch_invocations(mesh.indices, B.static_starts(mesh.num_tris, 12), "hash").sum())
        assert st["draws"] == 2 and st["invocations"] == 2 * inv
        del graph
    finally:
        gp.gp_destroy(ctx)
