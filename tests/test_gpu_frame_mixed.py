"""Frames that mix what writes the blocks' shared memory: naive, warp-voting and
group items write it with ordinary stores, the pipelines bulk-copy index windows
over it, and the end of an index buffer whose length is not a multiple of four
is again written by ordinary stores, in the middle of a run.  Index counts of every
remainder, every order of methods, outputs equal to the naive single draw's bit
for bit, over repeated launches."""
import numpy as np
import pytest

import meshgen as mg
from oracle import shading as S
from helpers_gp import draw_gpu, uniforms_for

pytestmark = pytest.mark.gpu

# (variant, mode, batch_indices, max_unique, threads per group)
METHODS = [("sort", 1, 0, 128, 256), ("naive", 0, 0, 0, 0), ("hash", 1, 0, 128, 256), ("warp", 0, 96, 0, 0),
           ("phash", 0, 192, 0, 256), ("hash", 0, 63, 0, 64), ("sort", 0, 255, 0, 256), ("hash", 1, 0, 128, 128)]


@pytest.mark.parametrize("count,seed", [(64, 1), (400, 2)])
def test_mixed_items(count, seed):
    import torch
    import paper_1805_08893_gb300 as gp
    rng = np.random.default_rng(seed)
    base = mg.geodesic_sphere(20, seed)
    uni, _ = uniforms_for(base, S.SHADER_MVP)
    verts = torch.from_numpy(base.vertices).cuda()
    ctx = gp.gp_create("hash", stream=torch.cuda.current_stream())
    try:
        descs, keep = [], []
        for k in range(count):
            T = int(rng.integers(1, 1200)) if k % 3 else 85 * (k % 4) + k % 4 + 1
            first = int(rng.integers(0, base.num_tris - T + 1))
            mesh = mg.Mesh(base.vertices, base.indices[3 * first: 3 * (first + T)].copy(), base.fmt, f"draw{k}")
            variant, mode, S_, nu, G = METHODS[int(rng.integers(0, len(METHODS)))]
            idx = torch.from_numpy(mesh.indices.view(np.int32).copy()).cuda()
            out = torch.empty(T * 21, device="cuda")
            keep.append((mesh, idx, out))
            descs.append(gp.draw_desc(idx, verts, gp.GP_SHADER_MVP, uni, out, variant=variant, mode=mode,
                                      batch_indices=S_, max_unique=nu, threads_per_group=G))
        want = [draw_gpu(mesh, "naive", S.SHADER_MVP, "static", uni, debug=False).out.reshape(-1)
                for mesh, _, _ in keep]
        frame = gp.gp_frame_create(ctx, descs)
        for _ in range(5):
            for _, _, out in keep:
                out.fill_(float("nan"))
            gp.gp_frame_submit(frame, ctx)
            assert gp.gp_sync(ctx, raise_on_error=False) == gp.GP_OK
            for k, (_, _, out) in enumerate(keep):
                assert np.array_equal(out.cpu().numpy().view(np.uint32), want[k].view(np.uint32)), k
        gp.gp_frame_destroy(frame)
    finally:
        gp.gp_destroy(ctx)
