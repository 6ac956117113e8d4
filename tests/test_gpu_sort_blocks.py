"""Sorting draws at the edges of the rule for their blocks: batches of as many
indices as threads and one triangle more, as many batches as two per SM and one
more, loads of 256 steps and one more, static and dynamic.  Outputs must equal the
naive kernel's bit for bit and the counts the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu

GRID = mg.grid_mesh(140)  # 38,642 triangles


@pytest.mark.parametrize("tris,S_,threads", [(304 * 85, 255, 256), (304 * 85 + 1, 255, 256), (30000, 258, 256),
                                             (304 * 42, 126, 128), (304 * 42 + 1, 126, 128), (20000, 129, 128),
                                             (30000, 255, 512), (5000, 24, 128), (30000, 48, 256)])
@pytest.mark.parametrize("shader,steps", [("mvp", 0), ("load", 256), ("load", 257)])
def test_static(tris, S_, threads, shader, steps):
    mesh = mg.Mesh(GRID.vertices, GRID.indices[: 3 * tris].copy(), GRID.fmt, "grid")
    sid = {"mvp": S.SHADER_MVP, "load": S.SHADER_LOAD}[shader]
    uni, _ = uniforms_for(mesh, sid, steps=steps)
    want = draw_gpu(mesh, "naive", sid, "static", uni)
    got = draw_gpu(mesh, "sort", sid, "static", uni, batch_indices=S_, threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
    assert np.array_equal(got.inv, B.unique_per_batch(mesh.indices, B.static_starts(tris, S_)))


@pytest.mark.parametrize("tris", [305 * 64 - 1, 305 * 64])
@pytest.mark.parametrize("max_tris,threads", [(64, 256), (85, 256), (86, 256), (42, 128)])
def test_dynamic(tris, max_tris, threads):
    mesh = mg.Mesh(GRID.vertices, GRID.indices[: 3 * tris].copy(), GRID.fmt, "grid")
    uni, _ = uniforms_for(mesh, S.SHADER_ENVELOPE)
    want = draw_gpu(mesh, "naive", S.SHADER_ENVELOPE, "static", uni)
    got = draw_gpu(mesh, "sort", S.SHADER_ENVELOPE, "dynamic", uni, max_unique=64, max_tris=max_tris,
                   threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
