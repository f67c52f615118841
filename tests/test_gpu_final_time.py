"""The final stage of a call for the bridges alone against the same phases run for the rooted forest: on a graph
that the reduction does not help it may not cost much more than they do."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _random(V, d, seed=0):
    rng = np.random.default_rng(int(1000 * d) + V + seed)
    return tuple(rng.integers(0, V, int(d * V)).astype(np.int32) for _ in range(2))


def _final_ms(cuda_lib, u, v, V, call):
    ctx = cuda_lib.Context(device="cuda:0", profile=True, ap_fused=-1)
    if V <= 4096:
        ctx.set_opts(ap_fused=-1, test_barrier_polls=1 << 24)  # the grid form also where one block would do
    du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    for _ in range(9):
        got = getattr(ctx, call)(du, dv, V)
    return sorted(t["final"] for t in ctx.stage_ms_history(8))[4], got


def _compare(cuda_lib, u, v, V, most):
    rooted, _ = _final_ms(cuda_lib, u, v, V, "articulation_points")  # two passes: every phase, and the sort
    alone, got = _final_ms(cuda_lib, u, v, V, "find")
    assert got.cpu().numpy().tolist() == oracle.dfs_bridges(u, v, V).tolist()
    assert alone < most * rooted, (alone, rooted)


@pytest.mark.parametrize("V", [300_000, 500_000])
def test_phases_have_their_cache(cuda_lib, V):
    """A sparse graph with cycles throughout takes the phases: 1.6 times as long when the stage asks for so much
    shared memory that the gathers have no L1."""
    _compare(cuda_lib, *_random(V, 1.5), V, 1.3)
