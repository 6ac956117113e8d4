"""Draw records and tickets: many draws in flight without a gp_sync, draws
refused in between, and a captured draw replayed.  A record has to be empty
when its draw starts (the reuse kernel claims batches from it), so a wrong one
shows in the counts or in the output."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import assert_attrs_close, uniforms_for

pytestmark = pytest.mark.gpu

SMALL = {"batch_indices": 12}  # more batches than resident blocks: the last ones are claimed from the record


def _buffers(mesh, torch):
    return (torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda(), torch.from_numpy(mesh.vertices).cuda(),
            torch.zeros(mesh.num_tris * 21, dtype=torch.float32, device="cuda"))


@pytest.mark.parametrize("draws", [1, 1023, 1024, 1025, 3000])
def test_more_draws_than_records(draws):
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = mg.grid_mesh(64)
    uni, ref = uniforms_for(mesh, S.SHADER_MVP)
    idx, verts, out = _buffers(mesh, torch)
    ctx = gp.gp_create("hash", stream=torch.cuda.current_stream(), **SMALL)
    try:
        for k in range(draws):
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
            if k % 500 == 7:  # a refused draw takes no record
                with pytest.raises(gp.GpError):
                    gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_SKIN, uni, out)
        st = gp.gp_stats(ctx)
        inv = int(B.batch_invocations(mesh.indices, B.static_starts(mesh.num_tris, 12), "hash").sum())
        assert st["draws"] == draws and st["invocations"] == draws * inv
        assert st["batches"] == draws * (len(B.static_starts(mesh.num_tris, 12)) - 1)
        assert_attrs_close(out.cpu().numpy().reshape(-1, 3, 7), S.draw(mesh, S.SHADER_MVP, ref), S.SHADER_MVP, mesh)
    finally:
        gp.gp_destroy(ctx)


def test_refused_inside_enqueue_gives_its_record_back():
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = mg.grid_mesh(64)
    uni, _ = uniforms_for(mesh, S.SHADER_MVP)
    idx, verts, out = _buffers(mesh, torch)
    ctx = gp.gp_create("hash", mode=gp.GP_BATCH_DYNAMIC, stream=torch.cuda.current_stream(), max_unique=12, max_tris=4)
    try:
        for k in range(40):
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
            with pytest.raises(gp.GpError):
                gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out, partition=99)
        st = gp.gp_stats(ctx)
        starts = B.dynamic_partition(mesh.indices, 12, 4, 4096)
        assert st["draws"] == 40
        assert st["invocations"] == 40 * int(B.batch_invocations(mesh.indices, starts, "hash").sum())
    finally:
        gp.gp_destroy(ctx)


def test_captured_draw_replays():
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = mg.grid_mesh(64)
    uni, ref = uniforms_for(mesh, S.SHADER_MVP)
    idx, verts, out = _buffers(mesh, torch)
    stream = torch.cuda.Stream()
    ctx = gp.gp_create("hash", stream=stream, **SMALL)
    try:
        with torch.cuda.stream(stream):
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
        gp.gp_sync(ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
        want = S.draw(mesh, S.SHADER_MVP, ref)
        for _ in range(3):
            out.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert_attrs_close(out.cpu().numpy().reshape(-1, 3, 7), want, S.SHADER_MVP, mesh)
        del graph
    finally:
        gp.gp_destroy(ctx)
