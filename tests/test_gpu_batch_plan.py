"""Batches planned on the device (256 graphs and more) against the same graphs in batches that the host plans; a tuned plan in calls that are waited for."""

import time

import numpy as np
import pytest
import torch

import graphgen
import oracle
import paper_2108_07346_gb300 as pb

pytestmark = pytest.mark.gpu

SIZES = [0, 1, 2, 3, 64, 700, 1024, 1025, 2000, 3008, 3009, 4096, 4097, 6000]


def results(ctx, u, v, off, Vs):
    out, counts, at = ctx.find_batched(u, v, off, Vs)
    out, counts = out.cpu().numpy(), counts.cpu().numpy()
    return [(int(c), out[a:a + 2 * max(int(c), 0)].tolist()) for c, a in zip(counts, at)]


@pytest.mark.parametrize("G", [256, 257, 1024, 1500])
@pytest.mark.parametrize("split", [0, 300])
def test_planned_on_device_equals_host(G, split):
    """Every class, empty graphs and lists, graphs above the shared-memory size among the others, lists cut in up
    to 64 parts, more graphs than the block has threads; one vertex id out of range."""
    rng = np.random.default_rng(G + split)
    Vs = np.array([SIZES[i % len(SIZES)] for i in range(G)], dtype=np.int32)
    us, vs = [], []
    for g, V in enumerate(Vs.tolist()):
        E = 0 if V < 2 or g % 17 == 5 else int(rng.integers(1, 5 * V))
        u, v = graphgen.random_multigraph(1000 * G + g, V, E) if E else (np.empty(0), np.empty(0))
        us.append(np.asarray(u, dtype=np.int32))
        vs.append(np.asarray(v, dtype=np.int32))
    us[4] = us[4].copy()
    us[4][-1] = 64  # SIZES[4] vertices
    off = np.concatenate([[0], np.cumsum([len(u) for u in us])]).astype(np.int64)
    u = torch.from_numpy(np.concatenate(us)).cuda()
    v = torch.from_numpy(np.concatenate(vs)).cuda()
    ctx = pb.Context()
    ctx.set_batch_split(split)
    got = results(ctx, u, v, off, Vs)
    assert results(ctx, u, v, off, Vs) == got  # the other staging copy
    want = []
    for a in range(0, G, 255):
        b = min(G, a + 255)
        want += results(ctx, u, v, off[a:b + 1], Vs[a:b])
    assert got == want
    assert got[4][0] < 0 and sum(c for c, _ in got) > 100


@pytest.mark.parametrize("large", [False, True])
def test_batches_behind_one_another(large):
    """A batch planned on the device, and behind it, not waited for, batches that the host plans (the last one is
    still running) and a single call, all on one context; then, idle again, one more of the first kind.  With and
    without graphs above the shared-memory size among them."""
    G = 400
    rng = np.random.default_rng(9)
    sizes = [5, 300, 1000, 2000, 4096] + ([5000] if large else [])
    Vs = rng.choice(sizes, G).astype(np.int32)
    us, vs = [], []
    for g, V in enumerate(Vs.tolist()):
        a, b = graphgen.random_multigraph(70_000 + g, V, int(rng.integers(V // 2, 40 * V)))
        us.append(np.asarray(a, dtype=np.int32))
        vs.append(np.asarray(b, dtype=np.int32))
    off = np.concatenate([[0], np.cumsum([len(a) for a in us])]).astype(np.int64)
    u, v = torch.from_numpy(np.concatenate(us)).cuda(), torch.from_numpy(np.concatenate(vs)).cuda()
    want = [oracle.dfs_bridges(a, b, V).tolist() for a, b, V in zip(us, vs, Vs.tolist())]

    def check(out, counts, at):
        out, counts = out.cpu().numpy(), counts.cpu().numpy()
        for g in range(G):
            assert out[at[g]:at[g] + 2 * counts[g]].reshape(-1, 2).tolist() == want[g]

    ctx = pb.Context()
    check(*ctx.find_batched(u, v, off, Vs))
    sets = [ctx.find_batched(u, v, off, Vs, sync=False) for _ in range(5)]
    g = int(np.argmax(Vs))
    single = ctx.find(u[off[g]:off[g + 1]], v[off[g]:off[g + 1]], int(Vs[g])).cpu().numpy().tolist()
    sets.append(ctx.find_batched(u, v, off, Vs, sync=False))
    torch.cuda.synchronize()
    assert single == want[g]
    for s in sets:
        check(*s)
    check(*ctx.find_batched(u, v, off, Vs))


def test_a_tuned_plan_is_no_slower_when_waited_for():
    """2,048 graphs of 300 to 500 vertices: a shorter prefix gains a few microseconds in batches enqueued behind one
    another, and costs the device's planning (120 us) where each batch is waited for."""
    G = 2048
    rng = np.random.default_rng(3)
    Vs = rng.integers(300, 500, G).astype(np.int32)
    Es = Vs.astype(np.int64) * (Vs - 1) // 4
    off = np.concatenate([[0], np.cumsum(Es)]).astype(np.int64)
    size = torch.from_numpy(np.repeat(Vs, Es)).cuda()
    u, v = (torch.randint(0, 1 << 30, size.shape, dtype=torch.int32, device="cuda").remainder_(size) for _ in range(2))
    ctx = pb.Context()

    def waited():
        out, counts, _ = ctx.find_batched(u, v, off, Vs)
        times = []
        for _ in range(21):
            t = time.perf_counter()
            ctx.find_batched(u, v, off, Vs, out=out, counts=counts)
            times.append(time.perf_counter() - t)
        return sorted(times)[10], counts.cpu().numpy()

    fresh, want = waited()
    ctx.batch_autotune(u, v, off, Vs)
    tuned, got = waited()
    assert np.array_equal(got, want)
    assert tuned < 1.25 * fresh
