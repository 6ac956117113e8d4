"""The sorting draws over the networks' sizes: 32-bit keys with 4 or 8 per
thread and other counts, 64-bit keys (a vertex buffer too large for 32), batches
that leave the network partly empty.  Ids ascend within a batch only inside the
kernel, so what shows is the output and the counts: they must equal the naive
kernel's and the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S_,threads", [(24, 32), (63, 64), (255, 64), (255, 128), (510, 128), (513, 128), (768, 256),
                                        (1023, 256), (1026, 256), (2046, 512), (1536, 128)])
@pytest.mark.parametrize("vertices", [1600, 5_000_000])
def test_sort_sizes(S_, threads, vertices):
    grid = mg.grid_mesh(40)
    verts = grid.vertices
    idx = grid.indices
    if vertices > 1600:  # ids beyond what 32-bit keys hold beside a position
        verts = np.zeros((vertices, 8), dtype=np.float32)
        verts[vertices - 1600:] = grid.vertices
        idx = (grid.indices + (vertices - 1600)).astype(np.uint32)
    mesh = mg.Mesh(verts, idx, mg.FMT_PNU32, "grid")
    uni, _ = uniforms_for(mesh, S.SHADER_MVP)
    want = draw_gpu(mesh, "naive", S.SHADER_MVP, "static", uni)
    got = draw_gpu(mesh, "sort", S.SHADER_MVP, "static", uni, batch_indices=S_, threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.ids, mesh.indices)
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
    assert np.array_equal(got.inv, B.unique_per_batch(mesh.indices, B.static_starts(mesh.num_tris, S_)))


@pytest.mark.parametrize("S_,threads", [(255, 64), (510, 128), (768, 256), (2046, 512)])
@pytest.mark.parametrize("steps", [640, 641])  # either side of the line past which half of the threads consume
def test_sort_load_steps(S_, threads, steps):
    mesh = mg.grid_mesh(40)
    uni, _ = uniforms_for(mesh, S.SHADER_LOAD, steps=steps)
    want = draw_gpu(mesh, "naive", S.SHADER_LOAD, "static", uni)
    got = draw_gpu(mesh, "sort", S.SHADER_LOAD, "static", uni, batch_indices=S_, threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
    assert np.array_equal(got.inv, B.unique_per_batch(mesh.indices, B.static_starts(mesh.num_tris, S_)))
