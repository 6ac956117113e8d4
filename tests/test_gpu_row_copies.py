"""The envelope shader with hashing on a grid: a vertex row's copy starts as soon as
its id is known, for every shader alike.  (Copied one per lane after the ids, the
batches of 64 triangles took 1.09 times as long, while MVP draws did not change.)"""
import numpy as np
import pytest

import meshgen as mg
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["hash", "phash"])
@pytest.mark.parametrize("mode,cfg", [("dynamic", {"max_unique": 64, "max_tris": 64}), ("static", {"batch_indices": 255}),
                                      ("dynamic", {"max_unique": 320, "max_tris": 426, "hash_slots": 2048})])
def test_envelope_rows(variant, mode, cfg):
    mesh = mg.grid_mesh(120)
    uni, _ = uniforms_for(mesh, S.SHADER_ENVELOPE)
    want = draw_gpu(mesh, "naive", S.SHADER_ENVELOPE, "static", uni)
    got = draw_gpu(mesh, variant, S.SHADER_ENVELOPE, mode, uni, **cfg)
    assert got.status == 0
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
