"""Static batches with rows for some of their vertices: draws large enough to run
that way (more batches than blocks with all the rows), whose batches hold more
unique vertices than there are rows, about as many, and fewer.  Outputs must equal
the naive kernel's bit for bit and the counts the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu

V = 6000


def _mesh(which, S_, batches):
    rng = np.random.default_rng(S_)
    n = batches * S_ - 3  # the last batch is short
    if which == "distinct":
        ids = np.concatenate([rng.permutation(V) for _ in range(-(-n // V))])[:n]
    else:  # about as many unique vertices as rows, from batch to batch more or fewer
        pool = rng.integers(S_ // 8, S_ // 2, size=batches)
        ids = np.concatenate([(b * 31 + rng.integers(0, p, size=S_)) % V for b, p in enumerate(pool)])[:n]
    return mg.Mesh(mg.random_vertices(1, V), ids.astype(np.uint32), mg.FMT_PNU32, which)


@pytest.mark.parametrize("which", ["distinct", "some"])
@pytest.mark.parametrize("variant,S_,threads", [("hash", 768, 256), ("phash", 768, 128), ("sort", 768, 256),
                                                ("hash", 192, 64), ("hash", 381, 64), ("phash", 1023, 512)])
@pytest.mark.parametrize("shader", ["mvp", "skin", "envelope"])
def test_rows_for_some(which, variant, S_, threads, shader):
    mesh, palette = _mesh(which, S_, 2500 if threads == 64 else 1300), None
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


def test_default_table_without_locality():
    """The default hash table is as fast as the one asked for by its size, where the batches fill it."""
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = _mesh("distinct", 768, 2000)
    uni, _ = uniforms_for(mesh, S.SHADER_MVP)
    idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
    verts = torch.from_numpy(mesh.vertices).cuda()
    out = torch.zeros(mesh.num_tris * 21, device="cuda")
    best = []
    for slots in (0, 2048):  # 2048: the documented default of 768 unique vertices
        ctx = gp.gp_create("hash", batch_indices=768, hash_slots=slots, stream=torch.cuda.current_stream())
        try:
            times = []
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(20):
                    gp.gp_submit_drawcall(ctx, idx, verts, gp.GP_SHADER_MVP, uni, out)
                b.record()
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
                gp.gp_sync(ctx)
            best.append(min(times))
        finally:
            gp.gp_destroy(ctx)
    assert best[0] < 1.15 * best[1]
