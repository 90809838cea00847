"""Residual counts of the surrogate at the sizes where the kernel's routes change, against a plain count."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _counts(g, pop):
    """(r0, r1, r2) by their definitions, from adjacency lists; a repeated gene counts the nodes whose
    first deleted neighbour it is once per repeat."""
    out = np.zeros((pop.shape[0], 3), dtype=np.int32)
    rp, col, deg = g.row_ptr, g.col, np.diff(g.row_ptr)
    src = np.repeat(np.arange(g.n), deg)
    for r, row in enumerate(pop):
        times = np.bincount(row[(row >= 0) & (row < g.n)], minlength=g.n)
        dead = times > 0
        gone = np.bincount(src, weights=dead[col], minlength=g.n).astype(np.int64)
        live = deg - gone
        for u in np.nonzero(~dead & (gone > 0) & (live <= 1))[0]:
            near = col[rp[u]:rp[u + 1]]
            weight = times[near[dead[near]][0]]
            out[r, live[u]] += weight
            if live[u] == 1:
                w = near[~dead[near]][0]
                out[r, 2] += weight * (live[w] == 1 and (u < w or gone[w] == 0))
    return out


# n around a bitmap word; 80000: 256 to 1024 threads per row by the number of rows; 700000: three
# bitmaps exceed shared memory.  Stars and paths hold the nodes of degree one and two.
@pytest.mark.parametrize("n,rows", [(31, 5), (33, 40), (1000, 700), (80000, 3), (80000, 640), (700000, 4)])
@pytest.mark.parametrize("shape", ["tree", "sparse", "hubs", "path"])
def test_residual_counts(n, rows, shape):
    import torch

    from paper_2412_20980_gb300 import Context, Surrogate, make_surrogate_config

    rng = np.random.default_rng(n + rows)
    if shape == "path":
        g = synth.named_graph("path", n)
    else:  # random recursive tree, or a sparse random graph over part of the nodes
        v = np.arange(1, n)
        u = (v * rng.random(n - 1)).astype(np.int64)
        if shape == "sparse":
            u, v = rng.integers(0, n, (2, int(1.3 * n)))
            u, v = u[u != v], v[u != v]
        g = synth.csr_from_edges(n, u, v)
    k = n // 5 if n <= 1000 else 2500
    few = min(rows, 12)
    pop = np.stack([rng.permutation(n)[:k] for _ in range(few)]).astype(np.int32)
    if shape == "hubs":
        top = np.argsort(-np.diff(g.row_ptr), kind="stable")[:k]
        for row in pop[::2]:  # hubs first, every gene once
            row[:] = np.concatenate([top[: k // 2], rng.permutation(np.setdiff1d(np.arange(n), top))[: k - k // 2]])
        pop[1::2, : k // 2] = np.stack([rng.permutation(top)[: k // 2] for _ in pop[1::2]])  # with repeated genes
    pop[0, :2] = (-1, n)  # ignored
    full = np.concatenate([pop] * (rows // few + 1))[:rows]
    with Context(0) as ctx:
        ctx.graph_upload(g.row_ptr, g.col)
        sg = Surrogate(ctx, make_surrogate_config(batch=16, ring=16), seed=1)
        got = sg.residual(torch.from_numpy(full).cuda()).cpu().numpy()
    want = _counts(g, pop)
    assert np.array_equal(got, np.concatenate([want] * (rows // few + 1))[:rows])
