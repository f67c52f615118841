"""The fused articulation stream's pair labels (one per F' component and class): many classes, few, more
classes than labels, one component split into many classes -- against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cliques,size,joined", [(2000, 5, False), (2000, 5, True), (11_000, 6, True), (30, 900, True),
                                                 (16_500, 6, False), (1, 3000, True)])
def test_many_classes(cuda_lib, cliques, size, joined):
    import torch

    rng = np.random.default_rng(cliques + size)
    V = cliques * size
    E = 9 * V + 8000  # past the sample: the stream meets every class
    c = rng.integers(0, cliques, E) * size
    u, v = c + rng.integers(0, size, E), c + rng.integers(0, size, E)
    if joined:  # a chain of cliques that share no edge: the joints are cut vertices
        a = np.arange(cliques - 1) * size
        u, v = np.concatenate([u, a, a + 1]), np.concatenate([v, a + size, a + size])
        order = rng.permutation(len(u))
        u, v = u[order], v[order]
    name = rng.permutation(V)
    u, v = name[u].astype(np.int32), name[v].astype(np.int32)
    ctx = cuda_lib.Context(device="cuda:0")
    du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    pts, br = ctx.articulation_points(du, dv, V, with_bridges=True)
    assert ctx.last_config()["ap_fused"] == 1
    assert np.array_equal(pts.cpu().numpy(), oracle.articulation_points(u, v, V))
    assert br.cpu().numpy().tolist() == oracle.dfs_bridges(u, v, V).tolist()
