"""K-means passes that reuse a tile's centroid list, and the ways a list or the candidates can overflow."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("shape,n_mu,iters,early", [
    ((12, 12, 12), 1500, 8, False),     # more candidates than shared memory holds, lists that never fit
    ((9, 11, 10), 300, 25, False),      # half tiles, ragged; short lists (few grid points per tile)
    ((33, 30, 37), 200, 60, False),     # full tiles after half, lists reused for many passes
    ((64, 57, 66), 90, 40, True),       # 8 x 8 x 8 tiles, early stop
])
def test_lists_match_oracle(shape, n_mu, iters, early):
    rng = np.random.default_rng(n_mu)
    n_r = int(np.prod(shape))
    w = rng.random(n_r) ** 3
    if not early:   # a point without weight may move without moving a centroid, which the early stop does not see
        w[rng.random(n_r) < 0.1] = 0.0
    cell = tuple(0.4 * s for s in shape)
    init = np.sort(rng.choice(n_r, n_mu, replace=False)).astype(np.int64)
    ref = O.kmeans(w, shape, cell, n_mu, init, iters, early_stop=early)
    got = isdf.kmeans(torch.from_numpy(w).to(DEV), shape, cell, n_mu, torch.from_numpy(init), iters, early_stop=early)
    assert np.array_equal(got["labels"].cpu().numpy(), ref["labels"])
    assert np.array_equal(got["centroids"].cpu().numpy(), ref["centroids"])
    assert np.array_equal(got["idx"].cpu().numpy(), ref["idx"])
    st = got["stats"].cpu().numpy()
    assert (st[0], st[1], st[2]) == (ref["n_iter"], ref["near_ties"], ref["empty"])
    J = got["objective"].cpu().numpy()
    assert np.allclose(J, ref["objective"], rtol=1e-12, atol=0)   # the bound of the other K-means tests


def test_captured_passes_repeat():
    """The chained launches inside a CUDA graph: a replay on other weights equals the eager call."""
    shape, cell, n_mu, iters = (30, 28, 27), (9.0, 8.4, 8.1), 120, 30
    g = torch.Generator(device=DEV).manual_seed(3)
    n_r = int(np.prod(shape))
    w0, w1 = (torch.rand(n_r, dtype=torch.float64, device=DEV, generator=g) + 0.01 for _ in range(2))
    init = torch.randperm(n_r, device=DEV, generator=g)[:n_mu].sort().values
    ws = torch.empty(isdf.kmeans_workspace_bytes(shape, n_mu), dtype=torch.uint8, device=DEV)
    w = w0.clone()
    isdf.kmeans(w, shape, cell, n_mu, init, iters, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = isdf.kmeans(w, shape, cell, n_mu, init, iters, workspace=ws)
    w.copy_(w1)
    graph.replay()
    torch.cuda.synchronize()
    ref = isdf.kmeans(w1, shape, cell, n_mu, init, iters)
    for k in ("idx", "labels", "centroids", "objective", "stats"):
        assert torch.equal(out[k], ref[k]), k


def test_more_candidates_than_shared_memory_holds():
    """2,048 centroids in 8 layers at one side of 64^3, on every second point of a layer, alone with weight: tiles opposite
    have up to 1,770 as candidates (whole 8 x 8 x 8 tiles; the own list of two warps in three overflows, of the others not),
    and points between two rows have equal distances."""
    n, x, y = 64, np.arange(2, 10), np.arange(16, 48, 2)
    init = ((x[:, None, None] * n + y[None, :, None]) * n + y[None, None, :]).reshape(-1).astype(np.int64)
    w = np.zeros(n ** 3)
    w[init] = 0.5 + np.random.default_rng(5).random(init.size)
    cell = (0.25 * n,) * 3
    ref = O.kmeans(w, (n,) * 3, cell, init.size, init, 2)
    got = isdf.kmeans(torch.from_numpy(w).to(DEV), (n,) * 3, cell, init.size, torch.from_numpy(init), 2)
    for k in ("labels", "centroids", "idx"):
        assert np.array_equal(got[k].cpu().numpy(), ref[k]), k
    st = got["stats"].cpu().numpy()
    assert (st[0], st[1], st[2]) == (ref["n_iter"], ref["near_ties"], ref["empty"]) and ref["near_ties"] > 100000
    bare = isdf.kmeans(torch.from_numpy(w).to(DEV), (n,) * 3, cell, init.size, torch.from_numpy(init), 2, objective=False)
    assert torch.equal(bare["labels"], got["labels"]) and torch.equal(bare["stats"], got["stats"])


def test_time_of_crowded_centroids():
    """Tiles that have thousands of candidates cost what their number asks for. 4,096 centroids in a ball of 14 spacings in
    128^3 against the same number all over the cell: 16 times the time when a candidate's coordinates are formed once a
    chunk, 149 times when they were formed at every use."""
    n, n_mu = 128, 4096
    g = torch.Generator(device=DEV).manual_seed(n_mu)
    ax = torch.arange(n, device=DEV, dtype=torch.float64) - 63.5
    ball = (ax[:, None, None] ** 2 + ax[None, :, None] ** 2 + ax[None, None, :] ** 2 <= 14.0 ** 2).reshape(-1)
    ms = []
    for inside in (torch.ones_like(ball), ball):
        w = inside * (0.5 + torch.rand(n ** 3, dtype=torch.float64, device=DEV, generator=g))
        at = inside.nonzero().reshape(-1)
        init = at[torch.randperm(at.numel(), device=DEV, generator=g)[:n_mu]].sort().values
        run = lambda: isdf.kmeans(w, (n,) * 3, (48.0,) * 3, n_mu, init, 10)   # noqa: E731
        run()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        run()
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    assert ms[1] < 90 * ms[0], ms
