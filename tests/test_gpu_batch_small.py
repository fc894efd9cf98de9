"""Batches of graphs of a few vertices each (a warp's 1,024 rows hold more than 32 graphs: a row a lane
in the reductions), alone and beside large ones, against the single-graph update in 64 bits."""
import numpy as np
import pytest
import torch

import paper_2605_07391_gb300 as mb

pytestmark = pytest.mark.gpu
ALPHA = 0.85


def _batch(sizes, seed):
    """Graphs of the given sizes: vertex i links to a few vertices of its graph, some to none."""
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    graph = np.repeat(np.arange(len(sizes)), sizes)
    deg = rng.integers(0, 5, n)
    src = np.repeat(np.arange(n), deg)
    dst = off[graph[src]] + (rng.random(src.size) * np.asarray(sizes)[graph[src]]).astype(np.int64)
    key = np.unique(dst * n + src)
    dst, src = key // n, key % n
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(dst, minlength=n), out=row_ptr[1:])
    out = np.bincount(src, minlength=n)
    return off, graph, row_ptr.astype(np.int32), dst, src, 1.0 / out[src], out == 0


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("sizes", ["ones", "twos", "three_to_forty", "32_a_chunk", "33_a_chunk", "mixed"])
def test_updates(cuda_device, dtype, sizes):
    rng = np.random.default_rng(5)
    size = {"ones": np.ones(5000), "twos": np.full(3001, 2), "three_to_forty": rng.integers(3, 41, 2000),
            "32_a_chunk": np.full(320, 32), "33_a_chunk": np.full(340, 31),
            "mixed": np.concatenate([np.full(700, 3), [40_000], np.full(900, 5), [7, 20_001, 1]])}[sizes].astype(np.int64)
    off, graph, row_ptr, dst, src, val, dangling = _batch(size, 3)
    n = int(off[-1])
    inv = 1.0 / size[graph]
    b = mb.Batch(torch.from_numpy(row_ptr).cuda(), torch.from_numpy(src.astype(np.int32)).cuda(), off)
    v = torch.from_numpy(val).to("cuda", dtype)
    # an update's rounding is at most a few units of the type, and shrinks by alpha per update
    tol = 20 * torch.finfo(dtype).eps / (1 - ALPHA)
    pi = inv.copy()
    for k in range(1, 7):
        old = pi
        mass = np.bincount(graph[dangling], pi[dangling], minlength=size.size)
        pi = ALPHA * np.bincount(dst, val * pi[src], minlength=n) + (ALPHA * mass + 1 - ALPHA)[graph] * inv
        if k not in (1, 2, 6):
            continue
        got, info = b.pagerank(v, ALPHA, tol=0.0, max_iter=k)
        assert np.abs(got.double().cpu().numpy() - pi).max() <= tol * pi.max()
        resid = np.bincount(graph, np.abs(pi - old), minlength=size.size)
        assert np.abs(info["resid"] - resid).max() <= tol


def test_time_of_tiny_graphs(cuda_device):
    """100,000 graphs of two vertices, 30 rounds: no warp goes through its graphs one by one (31 ms)."""
    size = np.full(100_000, 2, np.int64)
    off, _, row_ptr, _, src, val, _ = _batch(size, 3)
    b = mb.Batch(torch.from_numpy(row_ptr).cuda(), torch.from_numpy(src.astype(np.int32)).cuda(), off)
    v = torch.from_numpy(val).cuda().float()
    times = []
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        b.pagerank(v, ALPHA, tol=0.0, max_iter=30)
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    assert sorted(times)[2] < 12.0, times
