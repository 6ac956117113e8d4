"""Frames whose hash draws go through runs: batches of many draws, one after
another in the same pipeline, over chunks of items that end inside draws.
Draws of one triangle to several chunks, neighbours with different buffers,
uniforms, limits and shaders, some in groups instead of runs, one with an index
out of range.  Every output must equal the naive single draw's bit for bit, every
count the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu

# (mode, batch_indices, max_unique, threads per group)
LIMITS = [(1, 0, 256, 256), (1, 0, 128, 128), (0, 255, 0, 256), (1, 0, 64, 256), (0, 63, 0, 64), (0, 126, 0, 128)]


def _draws(count, seed, sizes):
    rng = np.random.default_rng(seed)
    base = mg.geodesic_sphere(20, seed)  # 8,000 triangles
    skin, palette = mg.skin_mesh(base, seed)
    for k in range(count):
        T = int(sizes[k % len(sizes)])
        shader = ["mvp", "skin", "envelope", "load"][int(rng.integers(0, 4))]
        src = skin if shader == "skin" else base
        first = int(rng.integers(0, base.num_tris - T + 1))
        mesh = mg.Mesh(src.vertices, src.indices[3 * first: 3 * (first + T)].copy(), src.fmt, f"draw{k}")
        sid = {"mvp": S.SHADER_MVP, "skin": S.SHADER_SKIN, "envelope": S.SHADER_ENVELOPE, "load": S.SHADER_LOAD}[shader]
        uni, _ = uniforms_for(mesh, sid, seed=k, palette=palette if shader == "skin" else None)
        variant = "phash" if rng.random() < 0.4 else "hash"
        yield mesh, sid, uni, variant, LIMITS[int(rng.integers(0, len(LIMITS)))]


@pytest.mark.parametrize("count,seed,sizes", [(1, 1, [1]), (3, 2, [1, 2, 3]), (60, 3, [1, 5, 85, 86, 400, 7]),
                                              (40, 4, [8000, 1, 3001, 256]), (300, 5, [2, 120])])
def test_runs_over_draws(count, seed, sizes):
    import torch
    import paper_1805_08893_gb300 as gp
    draws = list(_draws(count, seed, sizes))
    bad = 5 if count > 5 else None
    ctx = gp.gp_create("hash", stream=torch.cuda.current_stream())
    try:
        descs, keep = [], []
        for k, (mesh, sid, uni, variant, (mode, S_, nu, G)) in enumerate(draws):
            if k == bad:
                mesh.indices[1] = mesh.num_vertices
            idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
            verts = torch.from_numpy(mesh.vertices).cuda()
            out = torch.full((mesh.num_tris * 3 * gp.gp_out_floats(sid),), float("nan"), device="cuda")
            inv = torch.full((mesh.num_tris,), -1, dtype=torch.int32, device="cuda")
            keep.append((idx, verts, out, inv))
            descs.append(gp.draw_desc(idx, verts, sid, uni, out, None, inv, variant=variant, mode=mode,
                                      batch_indices=S_, max_unique=nu, threads_per_group=G))
        frame = gp.gp_frame_create(ctx, descs)
        for _ in range(2):
            for _, _, out, inv in keep:
                out.fill_(float("nan"))
                inv.fill_(-1)
            gp.gp_frame_submit(frame, ctx)
            status = gp.gp_sync(ctx, raise_on_error=False)
            assert status == (gp.GP_ERR_INDEX_RANGE if bad is not None else gp.GP_OK)
        st = gp.gp_stats(ctx)
        total = 0
        for k, ((mesh, sid, uni, variant, (mode, S_, nu, G)), (_, _, out, inv)) in enumerate(zip(draws, keep)):
            want = draw_gpu(mesh, "naive", sid, "static", uni, debug=False)
            got = out.cpu().numpy().reshape(want.out.shape)
            assert np.array_equal(got.view(np.uint32), want.out.view(np.uint32)), k
            starts = (B.static_starts(mesh.num_tris, S_) if mode == 0
                      else B.dynamic_partition(mesh.indices, nu, (4 * nu - 1) // 3, 4096))
            counts = B.unique_per_batch(mesh.indices, starts)
            if k != bad:
                assert np.array_equal(inv.cpu().numpy()[: len(counts)], counts), k
            total += int(counts.sum())
        if bad is None:
            assert st["invocations"] == 2 * total
        gp.gp_frame_destroy(frame)
    finally:
        gp.gp_destroy(ctx)
