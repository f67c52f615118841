"""Ordered compaction of the articulation points: one launch up to 64 tiles of 4,096 vertices, three above."""

import numpy as np
import pytest
import torch

import paper_2108_07346_gb300 as pb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [2, 3, 4095, 4096, 4097, 64 * 4096 - 1, 64 * 4096, 64 * 4096 + 1, 65 * 4096])
def test_caterpillar(V):
    """Even vertices form a path, each odd one hangs off the even one before it: the points are the even
    vertices that have a leaf (a path of two vertices has none)."""
    even, odd = np.arange(0, V, 2), np.arange(1, V, 2)
    u = np.concatenate([even[:-1], odd - 1]).astype(np.int32)
    v = np.concatenate([even[1:], odd]).astype(np.int32)
    want = odd - 1 if V > 2 else np.empty(0, np.int64)
    ctx = pb.Context()
    got = ctx.articulation_points(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), V)
    assert got.cpu().numpy().tolist() == want.tolist()
