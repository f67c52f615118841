"""The sampled certificate (sample.cu) at the sizes where it can go wrong: one and several edges a
thread, label and bitmap limits, lists certified whole and lists with a stream behind the sample,
long chains, hubs, parallel edges, lists sorted by their ends, unaligned starts -- against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _er(rng, V, E):
    return rng.integers(0, V, E).astype(np.int32), rng.integers(0, V, E).astype(np.int32)


def _check(pb, u, v, V, **opts):
    import torch

    du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    ctx = pb.Context(device="cuda:0", **opts)
    ref = oracle.dfs_bridges(u, v, V) if hasattr(oracle, "dfs_bridges") else oracle.bridges(u, v, V, 1)
    for _ in range(2):  # the second call finds the first one's workspace
        got = ctx.find(du, dv, V).cpu().numpy()
        assert got.tolist() == np.asarray(ref).reshape(-1, 2).tolist()
    cu, cv, ct = (t.cpu().numpy() for t in ctx.certificate(du, dv, V))
    # F spans what the list spans, F' lies inside F's sets, and neither holds a cycle
    comps = oracle.components(u, v, V)[1]
    assert int(ct.sum()) == V - len(np.unique(comps))
    f, f2 = (cu[ct], cv[ct]), (cu[~ct], cv[~ct])
    assert np.array_equal(oracle.components(f[0].copy(), f[1].copy(), V)[1], comps)
    c2 = oracle.components(f2[0].copy(), f2[1].copy(), V)[1]
    assert len(f2[0]) == V - len(np.unique(c2))


@pytest.mark.parametrize("V,E", [(1, 3), (2, 1), (33, 20), (1000, 999), (5000, 2 * (8 * 5000 + 4096)),
                                 (5000, 2 * (8 * 5000 + 4096) + 1), (20011, 900_001), (65_534, 400_000),
                                 (65_535, 1_300_000), (65_536, 1_300_001), (90_000, 3_000_000), (120_001, 2_500_000)])
def test_random_lists(cuda_lib, V, E):
    rng = np.random.default_rng(V * 7 + E)
    _check(cuda_lib, *_er(rng, V, E), V)


@pytest.mark.parametrize("V", [4097, 60_000, 130_000])
@pytest.mark.parametrize("shape", ["path", "reversed path", "star", "doubled path", "two hubs"])
def test_chains_and_hubs(cuda_lib, V, shape):
    x = np.arange(V - 1, dtype=np.int32)
    if shape == "path":
        u, v = x, x + 1
    elif shape == "reversed path":
        u, v = x[::-1].copy() + 1, x[::-1].copy()
    elif shape == "star":
        u, v = np.full(V - 1, V - 1, np.int32), x
    elif shape == "doubled path":
        u, v = np.concatenate([x, x + 1]), np.concatenate([x + 1, x])
    else:
        u = np.concatenate([np.full(V - 1, V - 1, np.int32), np.full(V - 1, V // 2, np.int32)])
        v = np.concatenate([x, x])
    _check(cuda_lib, u.astype(np.int32), v.astype(np.int32), V)


@pytest.mark.parametrize("V,E,warm", [(3000, 300_000, -1), (70_000, 2_000_000, -1), (70_000, 2_000_000, 5000),
                                      (3000, 300_000, 64), (130_000, 3_000_000, 200_000)])
def test_sorted_lists(cuda_lib, V, E, warm):
    rng = np.random.default_rng(E + warm)
    u, v = _er(rng, V, E)
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    order = np.lexsort((hi, lo))
    u, v = lo[order].copy(), hi[order].copy()
    u = np.concatenate([u, np.arange(V, V + 40, dtype=np.int32)])  # a pendant path at the end
    v = np.concatenate([v, np.arange(V - 1, V + 39, dtype=np.int32)])
    _check(cuda_lib, u, v, V + 40, warm_edges=warm)


@pytest.mark.parametrize("skip", [1, 2, 3])
def test_unaligned_slices(cuda_lib, skip):
    import torch

    rng = np.random.default_rng(skip)
    V, E = 2500, 200_003
    u, v = _er(rng, V, E)
    du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    got = cuda_lib.Context(device="cuda:0").find(du[skip:], dv[skip:], V).cpu().numpy()
    assert got.tolist() == oracle.bridges(u[skip:].copy(), v[skip:].copy(), V, 1).tolist()


@pytest.mark.parametrize("E,at", [(500, 499), (300_000, 0), (300_000, 299_999), (300_000, 150_001)])
def test_ids_out_of_range(cuda_lib, E, at):
    import torch

    rng = np.random.default_rng(at)
    V = 5000
    u, v = _er(rng, V, E)
    u[at] = V
    v[at] = V  # a loop out of range is an error all the same
    ctx = cuda_lib.Context(device="cuda:0")
    with pytest.raises(cuda_lib.BridgesError) as err:
        ctx.find(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), V)
    assert err.value.code == -2


@pytest.mark.parametrize("V", [9, 5000])
@pytest.mark.parametrize("warm", [1, 3, 7, 8, 9])
@pytest.mark.parametrize("E", [1, 2, 4, 7, 8, 9, 10, 16, 17])
def test_samples_below_one_group(cuda_lib, V, warm, E):
    """warm_edges below a sample's group of 8, lists around one and two groups: every edge is certified once, in
    each call that starts from a sample."""
    import torch

    rng = np.random.default_rng(100 * warm + E)
    x = np.arange(E, dtype=np.int32)
    paths = (x % (V - 1), x % (V - 1) + 1)  # (V 9, E 9 and more: a path with doubled edges)
    few = rng.integers(0, min(V, E + 1), (2, E)).astype(np.int32)
    for u, v in [tuple(a.astype(np.int32) for a in paths), (few[0].copy(), few[1].copy())]:
        _check(cuda_lib, u, v, V, warm_edges=warm)
        du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
        ref = oracle.dfs_bridges(u, v, V).tolist()
        count, labels = oracle.two_edge_components(u, v, V)
        ctx = cuda_lib.Context(device="cuda:0", warm_edges=warm)
        got, lab = ctx.two_edge_components(du, dv, V)
        assert got == count and np.array_equal(lab.cpu().numpy(), labels)
        points, bridges = ctx.articulation_points(du, dv, V, with_bridges=True)
        assert bridges.cpu().numpy().tolist() == ref
        assert points.cpu().numpy().tolist() == oracle.articulation_points(u, v, V).tolist()
        inc = cuda_lib.Incremental(device="cuda:0", warm_edges=warm)
        assert inc.reset(du, dv, V).cpu().numpy().tolist() == ref


@pytest.mark.parametrize("block", [1, 33, 100, 500, 1000])
@pytest.mark.parametrize("V,E", [(5000, 200_000), (70_000, 2_000_000), (130_000, 400_000)])
def test_blocks_of_odd_sizes(cuda_lib, block, V, E):
    """A block size that is no whole number of warps: labels, bitmap and (the second call) no snapshot."""
    rng = np.random.default_rng(block)
    u, v = _er(rng, V, E)
    _check(cuda_lib, u, v, V, block=block)
    _check(cuda_lib, u, v, V, block=block, warm_edges=0)


@pytest.mark.parametrize("V", [20_000, 53_000, 60_000, 130_000])
def test_long_unaligned_slices(cuda_lib, V):
    """A list long enough for interleaved tiles whose arrays start off a 16-byte boundary: the planted bridges and
    cut vertices of the aligned copy, in a time of the same order (one block alone would take 200 times as long)."""
    import time

    import torch

    E = 60_000_000
    gen = torch.Generator(device="cuda").manual_seed(V)
    u = torch.randint(0, V, (E + 1,), dtype=torch.int32, device="cuda", generator=gen)
    v = torch.randint(0, V, (E + 1,), dtype=torch.int32, device="cuda", generator=gen)
    tail = torch.arange(V, V + 40, dtype=torch.int32, device="cuda")  # a pendant path
    u[E - 40:E], v[E - 40:E] = tail, tail - 1
    u, v = u[:E], v[:E]
    ctx = cuda_lib.Context(device="cuda:0", ap_fused=0 if V != 60_000 else -1)

    def timed(call):
        call()
        torch.cuda.synchronize()
        t = time.perf_counter()
        got = call()
        torch.cuda.synchronize()
        return got.cpu().numpy().tolist(), time.perf_counter() - t

    path = list(range(V - 1, V + 39))  # (the rest, some 1,000 edges a vertex, has no bridge and no cut vertex)
    for call, want in ((ctx.find, [[x, x + 1] for x in path]), (ctx.articulation_points, path)):
        got, aligned = timed(lambda: call(u[4:], v[4:], V + 40))
        assert got == want
        got, unaligned = timed(lambda: call(u[1:], v[1:], V + 40))
        assert got == want
        assert unaligned < 8 * aligned


@pytest.mark.parametrize("V", [4097, 20_000, 37_147, 46_000, 49_527, 49_528, 53_000, 57_343, 57_344, 60_000, 99_000,
                               113_000, 130_000, 792_000, 793_000, 850_000, 917_400, 917_600, 1_500_000])
@pytest.mark.parametrize("opts", [{}, {"block": 1024}, {"block": 768}, {"block": 256}, {"M": 3}])
def test_stream_in_one_wave(cuda_lib, V, opts):
    """Every block of the automatic stream is resident at once, around the sizes at which the snapshot, with and
    without the winners' staging, fits an SM twice; and the result there."""
    import torch

    gen = torch.Generator(device="cuda").manual_seed(V)
    E = max(20 * V, 6_000_000)  # every partition has a snapshot, and every block edges
    u = torch.randint(0, V, (E,), dtype=torch.int32, device="cuda", generator=gen)
    v = torch.randint(0, V, (E,), dtype=torch.int32, device="cuda", generator=gen)
    tail = torch.arange(V, V + 40, dtype=torch.int32, device="cuda")  # a pendant path, its last edge doubled
    u[-41:], v[-41:] = torch.cat([tail, tail[-1:]]), torch.cat([tail - 1, tail[-1:] - 1])
    ctx = cuda_lib.Context(device="cuda:0", **opts)
    got = ctx.find(u, v, V + 40).cpu().numpy()
    cfg = ctx.last_config()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert 1 <= cfg["M"] * cfg["blocks_per_partition"] <= sms * cfg["stream_resident"]
    if V <= 850_000:  # (a sparse random graph has bridges of its own)
        want = [[V - 1 + i, V + i] for i in range(39)]
        inner = got[got[:, 1] < V]
        assert got[got[:, 1] >= V].tolist() == want and (V > 113_000 or len(inner) == 0)


@pytest.mark.parametrize("V", [60_000, 100_000])
def test_sparse_lists_take_one_another_s_time(cuda_lib, V):
    """Sparse random lists around the densities at which F and F' form their large sets: the sample's time changes
    little from one to the next (three to four times the others' when its last edges link before their sets meet)."""
    import torch

    gen = torch.Generator(device="cuda").manual_seed(V)
    times = {}
    for d in (0.85, 0.95, 1.05, 1.15, 1.5, 1.85, 1.95, 2.05, 2.15, 2.5):
        u, v = (torch.randint(0, V, (int(d * V),), dtype=torch.int32, device="cuda", generator=gen) for _ in range(2))
        ctx = cuda_lib.Context(device="cuda:0", profile=True)
        for _ in range(9):
            got = ctx.find(u, v, V)
        times[d] = sorted(t["warmup"] for t in ctx.stage_ms_history(8))[4]
        assert got.cpu().numpy().tolist() == oracle.dfs_bridges(u.cpu().numpy(), v.cpu().numpy(), V).tolist()
    assert max(times.values()) < 2 * sorted(times.values())[len(times) // 2], times


@pytest.mark.parametrize("V,opts", [(3000, {"warm_edges": 0}), (60_000, {"warm_edges": 0}), (130_000, {}),
                                    (500_000, {})])
def test_grid_of_a_list_that_links_edge_by_edge(cuda_lib, V, opts):
    """Without a sample every edge, or most of them, take the union-finds: a short list has as many blocks as a long
    one, and without a snapshot as many as four per SM."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    grids = set()
    for E in (20_000, 200_000, 3_000_000):
        rng = np.random.default_rng(E)
        u, v = _er(rng, V, E)
        du, dv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
        ctx = cuda_lib.Context(device="cuda:0", **opts)
        assert ctx.find(du, dv, V).cpu().numpy().tolist() == oracle.dfs_bridges(u, v, V).tolist()
        grids.add(ctx.last_config()["blocks_per_partition"])
    assert len(grids) == 1
    assert not opts or grids == {4 * sms}


def test_bitmap_of_nothing_halves_the_grid(cuda_lib):
    """Sparse random lists on more vertices than labels, whose prefix leaves F' without a large component: the
    automatic pass takes about the time of one block of 512 per SM (1.6 times it on the whole grid)."""
    import torch

    total = {}
    for V in (120_000, 160_000, 200_000):
        for d in (4, 6, 20):
            gen = torch.Generator(device="cuda").manual_seed(V + d)
            u, v = (torch.randint(0, V, (d * V,), dtype=torch.int32, device="cuda", generator=gen) for _ in range(2))
            found = []
            for name, opts in (("auto", {}), ("half", {"ctas_per_sm": 1, "block": 512})):
                ctx = cuda_lib.Context(device="cuda:0", profile=True, **opts)
                for _ in range(9):
                    got = ctx.find(u, v, V)
                total[name] = total.get(name, 0) + sorted(t["forest"] for t in ctx.stage_ms_history(8))[4]
                found.append(got.cpu().numpy().tolist())
            assert found[0] == found[1] == oracle.dfs_bridges(u.cpu().numpy(), v.cpu().numpy(), V).tolist()
    assert total["auto"] < 1.4 * total["half"], total
