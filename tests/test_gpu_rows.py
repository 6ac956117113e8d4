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
