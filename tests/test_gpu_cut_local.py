"""The cut-local kernel against the oracle where its layout, lists and fallbacks change."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2412_20980_gb300 import Context
    from paper_2412_20980_gb300 import build as b

    b.build()
    with Context(0) as c:
        yield c


def _graph(shape, n):
    rng = np.random.default_rng(n)
    if shape in ("star", "path"):
        return synth.named_graph(shape, n)
    v = np.arange(1, n)
    if shape == "tree":  # deletions shatter it: lists beyond a quarter of the graph
        return synth.csr_from_edges(n, (v * rng.random(n - 1)).astype(np.int64), v)
    if shape == "er":  # single nodes and many small components
        u, w = rng.integers(0, n, (2, int(0.9 * n)))
        return synth.csr_from_edges(n, u[u != w], w[u != w])
    back = np.concatenate([(v * rng.random(n - 1) ** 3).astype(np.int64) for _ in range(3)])  # low ids are hubs
    return synth.csr_from_edges(n, back, np.concatenate([v, v, v]))


# label and bitmap words, 256 / 512 / 1024 threads, one to eight members per SM, the largest ids
@pytest.mark.parametrize("n", [2, 3, 17, 33, 64, 1024, 1025, 2049, 5009, 20001, 33000, 56001])
@pytest.mark.parametrize("shape", ["star", "path", "tree", "er", "hubs"])
@pytest.mark.parametrize("objective", ["pc", "mcn"])
def test_cut_local_matches_oracle(ctx, n, shape, objective):
    import torch

    from paper_2412_20980_gb300.gapa import FITNESS_TREE_LOCAL, OBJECTIVE_MCN, OBJECTIVE_PC

    g = _graph(shape, n)
    rng = np.random.default_rng(7 * n)
    order = np.argsort(-g.degrees(), kind="stable").astype(np.int32)
    ctx.graph_upload(g.row_ptr, g.col)
    ctx.set_fitness_kernel(FITNESS_TREE_LOCAL)
    ctx.set_objective(OBJECTIVE_MCN if objective == "mcn" else OBJECTIVE_PC)
    try:
        for k, s in [(0, 2), (n // 20, 160), (n // 5, 12), (n - 1, 2), (n, 1)]:  # s: ordered members or not
            pop = np.stack([rng.permutation(n)[:k] for _ in range(s)]).astype(np.int32)
            for i in range(0, s, 3):
                h = k * (i % 7) // 6  # up to all of the genes among the hubs
                pop[i, :h] = order[:h]
                rest = order[h:]
                pop[i, h:] = rest[rng.permutation(rest.size)[:k - h]]
            if k > 3 and s > 1:
                pop[1, 2] = pop[1, 0]  # a repeated gene
            want = oracle.fitness(g.row_ptr, g.col, pop, "mcn" if objective == "mcn" else "bfs", nthreads=oracle.max_threads())
            got = ctx.fitness(torch.from_numpy(pop).cuda())
            ctx.sync()
            assert np.array_equal(got.cpu().numpy(), want), (k, s)
    finally:
        ctx.set_fitness_kernel(0)
        ctx.set_objective(OBJECTIVE_PC)
