"""Warp voting where a warp takes several batches one after another, with their
indices read ahead (up to 256 of them) and without: batch sizes at both sides of the
lines, every shader, ragged ends.  Outputs must equal the naive kernel's bit for
bit."""
import numpy as np
import pytest

import meshgen as mg
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu

GRID = mg.grid_mesh(120)  # 28,322 triangles
SHADERS = {"mvp": S.SHADER_MVP, "skin": S.SHADER_SKIN, "envelope": S.SHADER_ENVELOPE, "load": S.SHADER_LOAD}


@pytest.mark.parametrize("S_,threads", [(96, 64), (99, 64), (255, 64), (255, 256), (258, 64), (384, 256)])
@pytest.mark.parametrize("shader", list(SHADERS))
def test_many_batches_per_warp(S_, threads, shader):
    indices = np.concatenate([np.roll(GRID.indices.reshape(-1, 3), 7 * k, axis=0) for k in range(20)]).reshape(-1)
    mesh, palette = mg.Mesh(GRID.vertices, indices[:-3].copy(), GRID.fmt, "grids"), None
    if shader == "skin":
        mesh, palette = mg.skin_mesh(mesh, 3)
    uni, _ = uniforms_for(mesh, SHADERS[shader], palette=palette)
    want = draw_gpu(mesh, "naive", SHADERS[shader], "static", uni, debug=False)
    got = draw_gpu(mesh, "warp", SHADERS[shader], "static", uni, debug=False, batch_indices=S_,
                   threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
