"""The autotuner picks a plan by timing; tuned results stay exact; the JSON cache round-trips."""
import numpy as np
import pytest
import torch

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def test_autotune_and_cache(cuda_lib, tmp_path):
    from paper_2108_07346_gb300 import autotune

    g = graphgen.workload("mid")
    u = torch.from_numpy(np.array(g.u)).cuda()
    v = torch.from_numpy(np.array(g.v)).cuda()
    ctx = cuda_lib.Context(device="cuda:0")
    path = str(tmp_path / "tune.json")
    plan, hit = autotune.tune(ctx, u, v, g.V, path=path, reps=2)
    assert not hit and plan["M"] >= 1 and plan["us_per_call"] > 0
    got = ctx.find(u, v, g.V).cpu().numpy()
    assert ctx.last_config()["M"] == plan["M"]
    assert got.tolist() == oracle.bridges(g.u, g.v, g.V, 16).tolist()
    ctx2 = cuda_lib.Context(device="cuda:0")
    plan2, hit2 = autotune.tune(ctx2, u, v, g.V, path=path)
    assert hit2 and plan2 == plan
    assert ctx2.find(u, v, g.V).cpu().numpy().tolist() == got.tolist()


@pytest.mark.parametrize("V,E", [(500, 2_000), (4000, 20_000), (30_000, 40_000)])
def test_identical_candidates_keep_the_automatic_plan(cuda_lib, V, E):
    """Lists that one kernel, or one sample, certifies whole: no choice of a single partition changes what runs,
    and several partitions cost more, so nothing can beat the automatic plan but noise."""
    u, v = (torch.from_numpy(a).cuda() for a in graphgen.random_multigraph(V, V, E))
    ctx = cuda_lib.Context(device="cuda:0")
    for _ in range(3):
        plan = ctx.autotune(u, v, V)
        assert (plan["M"], plan["warm_edges"], plan["block"], plan["warm_block"]) == (1, -1, 0, 0)


def test_a_sampled_plan_keeps_no_warm_block(cuda_lib):
    """The block size of a launch that the plan does not have is not tuned; and a failed tuning leaves the
    options as they were."""
    g = graphgen.workload("mid")
    u = torch.from_numpy(np.array(g.u)).cuda()
    v = torch.from_numpy(np.array(g.v)).cuda()
    ctx = cuda_lib.Context(device="cuda:0")
    plan = ctx.autotune(u, v, g.V, reps=2)
    assert plan["M"] > 1 or plan["warm_block"] == 0
    small = cuda_lib.Context(device="cuda:0", workspace_bytes=1 << 20)
    opts = small.get_opts()
    with pytest.raises(cuda_lib.BridgesError):
        small.autotune(u, v, g.V)
    assert small.get_opts() == opts
