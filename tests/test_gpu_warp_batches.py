"""Warp voting at the edges of its two output paths: batches that are staged
whole and leave in one bulk store (at most 96 indices, starting and ending on
16-byte boundaries), batches written round by round, ragged last batches,
rounds of more than 32 corners.  Outputs must equal the naive kernel's bit for
bit, the counts the oracle's."""
import numpy as np
import pytest

import meshgen as mg
from oracle import batching as B
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu

GRID = mg.grid_mesh(40)  # 3,042 triangles


def _mesh(kind, tris):
    if kind == "grid":
        idx = GRID.indices
    elif kind == "equal":  # one round takes a whole batch
        idx = np.full(3 * 2000, 7, dtype=np.uint32)
    else:  # no repeats: ten triangles a round
        idx = np.concatenate([np.random.default_rng(k).permutation(1599) for k in range(4)]).astype(np.uint32)
    return mg.Mesh(GRID.vertices, idx[: 3 * tris].copy(), mg.FMT_PNU32, kind)


@pytest.mark.parametrize("kind,tris", [("grid", 3042), ("grid", 1), ("grid", 1021), ("equal", 1999), ("distinct", 1777)])
@pytest.mark.parametrize("S_,threads", [(3, 64), (9, 32), (12, 256), (48, 64), (93, 64), (96, 64), (96, 256), (99, 96),
                                        (384, 128)])
@pytest.mark.parametrize("shader", ["mvp", "envelope"])
def test_warp_batches(kind, tris, S_, threads, shader):
    mesh = _mesh(kind, tris)
    sid = S.SHADER_MVP if shader == "mvp" else S.SHADER_ENVELOPE
    uni, _ = uniforms_for(mesh, sid)
    want = draw_gpu(mesh, "naive", sid, "static", uni)
    got = draw_gpu(mesh, "warp", sid, "static", uni, batch_indices=S_, threads_per_group=threads)
    assert got.status == 0
    assert np.array_equal(got.ids, mesh.indices)
    assert np.array_equal(got.out.view(np.uint32), want.out.view(np.uint32))
    assert np.array_equal(got.inv, B.batch_invocations(mesh.indices, B.static_starts(mesh.num_tris, S_), "warp"))
