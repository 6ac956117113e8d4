"""Several draws folded together: the error returned is the worst of theirs, in
whatever order they failed."""
import numpy as np
import pytest

import meshgen as mg
from oracle import shading as S
from helpers_gp import uniforms_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", ["range", "stall"])
@pytest.mark.parametrize("by", ["submit", "sync"])
def test_worst_error_of_a_fold(first, by):
    import torch
    import paper_1805_08893_gb300 as gp
    mesh = mg.grid_mesh(8)
    uni, _ = uniforms_for(mesh, S.SHADER_MVP)
    idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
    bad = idx.clone()
    bad[0] = mesh.num_vertices  # out of range: drawn as zeros and reported
    verts = torch.from_numpy(mesh.vertices).cuda()
    out = torch.zeros(mesh.num_tris * 21, device="cuda")
    ctx = gp.gp_create("hash", stream=torch.cuda.current_stream())
    try:
        def draw(i):
            gp.gp_submit_drawcall(ctx, i, verts, gp.GP_SHADER_MVP, uni, out)

        def stall():  # a bounded wait runs out (~0.8 s) and is reported
            gp.gp_test_inject(ctx, gp.GP_TEST_STALL_WINDOW, 1)
            draw(idx)

        for f in ([lambda: draw(bad), stall] if first == "range" else [stall, lambda: draw(bad)]):
            f()
        for _ in range(1022):  # 1,024 draws in flight: the next one folds the completed ones
            draw(idx)
        torch.cuda.synchronize()
        with pytest.raises(gp.GpError) as e:
            if by == "submit":
                draw(idx)
            else:
                gp.gp_sync(ctx)
        assert e.value.status == gp.GP_ERR_TIMEOUT
        assert "GP_ERR_TIMEOUT" in gp.gp_last_error(ctx)
        assert gp.gp_stats(ctx)["draws"] == 1024
        draw(idx)
        assert gp.gp_sync(ctx) == gp.GP_OK
    finally:
        gp.gp_destroy(ctx)
