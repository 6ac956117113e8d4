"""The random walk on fields with empty cells: agents whose nearest eight cells are
all active, some, none, beside each other in a warp, with activity near and with none
in reach.  Positions must equal the oracle's bit for bit, and a step on a large
field with few active cells may not cost more than a step that is not bounded at
all (a captured call looks at every candidate)."""
import numpy as np
import pytest

import meshgen as mg
from oracle import walk as W

pytestmark = pytest.mark.gpu


def _run(act, keys, steps, variant):
    import torch
    import paper_1805_08893_gb300 as gp
    pos = torch.from_numpy(keys.view(np.int32).copy()).cuda()
    cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
    gp.gp_random_walk(torch.from_numpy(act.view(np.int32)).cuda(), pos, torch.empty_like(pos), cnt, steps, 9, variant,
                      batch_agents=96, threads=64)
    torch.cuda.synchronize()
    assert int(cnt[2]) == 0
    return pos.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("share", [0.002, 0.05, 0.3, 0.8, 0.97])
@pytest.mark.parametrize("width,height", [(17, 19), (70, 41), (300, 200)])
def test_share_of_active_cells(share, width, height):
    rng = np.random.default_rng(int(1000 * share) + width)
    act = np.where(rng.random((height, width)) < share, rng.integers(1, 1 << 20, size=(height, width)), 0).astype(np.uint32)
    act[: height // 3, : width // 2] = 0  # nothing in reach
    keys = mg.walk_agents(3, 300, width, height)
    want, _ = W.run(act, keys, 2, 9)
    for variant in ("naive", "hash", "sort", "warp"):
        assert np.array_equal(_run(act, keys, 2, variant), want), variant


def test_cost_on_a_sparse_field():
    import torch
    import paper_1805_08893_gb300 as gp
    g = torch.Generator(device="cuda").manual_seed(1)
    w = h = 4096
    n = 500_000
    act = ((torch.rand(h, w, generator=g, device="cuda") < 0.002).int() * 4096).contiguous()
    start = (torch.randint(0, w, (n,), generator=g, device="cuda") << 16
             | torch.randint(0, h, (n,), generator=g, device="cuda")).int()
    pos, scratch = start.clone(), torch.empty_like(start)
    cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
    stream = torch.cuda.Stream()

    def call():
        gp.gp_random_walk(act, pos, scratch, cnt, 4, 5, "naive", stream=stream)

    with torch.cuda.stream(stream):
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            call()

        def best(f):
            times = []
            for _ in range(5):
                pos.copy_(start)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                f()
                b.record(stream)
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
            return min(times)

        # row by row both, and the bounds of 4096 x 4096 cells once per call: at most a tenth of four steps
        assert best(call) < 1.3 * best(graph.replay)
    del graph
