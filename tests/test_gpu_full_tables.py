"""Hash tables with no slot to spare: batches of as many unique vertices as the
table has slots, so that the last ids probe far, over both ways in which a thread's
collided positions go on.  Outputs must equal the naive kernel's bit for bit and
the counts the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["hash", "phash"])
@pytest.mark.parametrize("shader", ["mvp", "envelope"])
@pytest.mark.parametrize("slots", [256, 512])
def test_full_table(variant, shader, slots):
    mesh = mg.Mesh(mg.random_vertices(1, 5000), mg.random_indices(3, 6000, 5000), mg.FMT_PNU32, "random")
    sid = {"mvp": S.SHADER_MVP, "envelope": S.SHADER_ENVELOPE}[shader]
    uni, _ = uniforms_for(mesh, sid)
    want = draw_gpu(mesh, "naive", sid, "static", uni)
    got = draw_gpu(mesh, variant, sid, "dynamic", uni, max_unique=slots, max_tris=400, hash_slots=slots,
                   threads_per_group=256)
    assert got.status == 0
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
    starts = B.dynamic_partition(mesh.indices, slots, 400, 4096)
    assert np.array_equal(got.inv, B.unique_per_batch(mesh.indices, starts))
