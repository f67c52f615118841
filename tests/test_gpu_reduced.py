"""The bridges of the reduced graph (F' components contracted) in each of its forms -- a forest, stripped
leaves, a core in shared memory, a core on the grid, a graph too cyclic to be reduced -- at the sizes
around their limits, and what reads its per-edge result (2-edge-connected components, incremental sets),
against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _dense(rng, V, E):
    return rng.integers(0, V, E), rng.integers(0, V, E)


def _build(shape, V, rng):
    """(u, v, V) of a graph of about V vertices; numbers are shuffled by the caller."""
    x = np.arange(V - 1)
    if shape == "cycle":
        return np.append(x, V - 1), np.append(x + 1, 0)
    if shape == "necklace":  # triangles joined by single edges
        k = V // 3
        a = 3 * np.arange(k)
        return (np.concatenate([a, a + 1, a + 2, a[:-1]]), np.concatenate([a + 1, a + 2, a, a[1:] + 1]))
    if shape == "ladder with tails":  # a long cycle band, a tail of 3 on every rung: stripped leaves, large core
        k = V // 5
        a = np.arange(k)
        t = 2 * k + 3 * a
        return (np.concatenate([a[:-1], k + a[:-1], a, a, t, t + 1]),
                np.concatenate([a[1:], k + a[1:], k + a, t, t + 1, t + 2]))
    if shape == "pendants":  # a dense core, pendant paths of up to 9, one long path
        core = max(8, V // 4)
        u, v = _dense(rng, core, 12 * core)
        y = core + np.arange(V - core)
        up = np.where(rng.random(V - core) < 0.2, rng.integers(0, core, V - core), y - 1)
        return np.concatenate([u, y]), np.concatenate([v, up])
    if shape == "two cores in a ring":  # cycles through single edges between dense parts, and pendants
        core = max(2, V // 64)
        us, vs = [], []
        for i in range(16):
            u, v = _dense(rng, core, 10 * core)
            us += [u + i * core, [i * core]]
            vs += [v + i * core, [((i + 1) % 16) * core + 1]]
        y = 16 * core + np.arange(V - 16 * core)
        us.append(y)
        vs.append(rng.integers(0, 16 * core, y.shape[0]))
        return np.concatenate(us), np.concatenate(vs)
    if shape == "star of leaves":
        u, v = _dense(rng, 50, 600)
        return np.concatenate([u, np.arange(50, V)]), np.concatenate([v, np.zeros(V - 50, np.int64)])
    return _dense(rng, V, int(1.4 * V))  # sparse random


SHAPES = ["cycle", "necklace", "ladder with tails", "pendants", "two cores in a ring", "star of leaves", "random"]


@pytest.mark.parametrize("V", [60, 1025, 4096, 4097, 16_500, 70_001])
@pytest.mark.parametrize("shape", SHAPES)
def test_bridges_and_components(cuda_lib, shape, V):
    import torch

    rng = np.random.default_rng(len(shape) * 1009 + V)
    u, v = _build(shape, V, rng)
    name = rng.permutation(V)
    u, v = name[u].astype(np.int32), name[v].astype(np.int32)
    order = rng.permutation(len(u))
    u, v = u[order], v[order]
    du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    ref = oracle.dfs_bridges(u, v, V).tolist()
    ctx = cuda_lib.Context(device="cuda:0")
    assert ctx.find(du, dv, V).cpu().numpy().tolist() == ref
    assert ctx.find(du, dv, V, 3).cpu().numpy().tolist() == ref
    ctx.set_opts(test_barrier_polls=1 << 24)  # the grid form also where one block would do
    assert ctx.find(du, dv, V).cpu().numpy().tolist() == ref
    ctx.set_opts()
    count, labels = oracle.two_edge_components(u, v, V)
    got, lab = ctx.two_edge_components(du, dv, V)
    assert got == count and np.array_equal(lab.cpu().numpy(), labels)
    inc = cuda_lib.Incremental(device="cuda:0")
    half = len(u) // 2
    inc.reset(du[:half], dv[:half], V)
    assert inc.add(du[half:], dv[half:]).cpu().numpy().tolist() == ref
    got, lab = inc.two_edge_components()
    assert got == count and np.array_equal(lab.cpu().numpy(), labels)
