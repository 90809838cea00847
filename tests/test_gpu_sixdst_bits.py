"""SixDST by bit rows against the dense reference and the dense products (whole numbers: bit-exact)."""
import numpy as np
import pytest

import synth
from oracle import sixdst_ref as sx

pytestmark = pytest.mark.gpu

AUTO, BITS, TMA = 4, 5, 3


@pytest.fixture(scope="module")
def ctx():
    from paper_2412_20980_gb300 import Context
    from paper_2412_20980_gb300 import build as b

    b.build()
    with Context(0) as c:
        yield c


def _fit(ctx, g, pop, hops, objective, kernel):
    import torch

    from paper_2412_20980_gb300.gapa import OBJECTIVE_SIXDST_MCN, OBJECTIVE_SIXDST_PC

    ctx.graph_upload(g.row_ptr, g.col)
    ctx.set_objective(OBJECTIVE_SIXDST_MCN if objective == "mcn" else OBJECTIVE_SIXDST_PC)
    ctx.set_sixdst_hops(hops)
    ctx.set_sixdst_kernel(kernel)
    out = ctx.fitness(torch.from_numpy(np.ascontiguousarray(pop, dtype=np.int32)).cuda())
    ctx.sync()
    return out.cpu().numpy()


# word and strip edges (32 and 128 columns), adjacencies below and above the whole-warp length
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 127, 128, 129, 257, 1025])
@pytest.mark.parametrize("hops", [1, 4, 7])
@pytest.mark.parametrize("objective", ["pc", "mcn"])
def test_bits_match_dense_reference(ctx, n, hops, objective):
    g = synth.named_graph("star", n) if n in (2, 257) else (
        synth.ba_graph(n, 2, n) if n > 4 else synth.csr_from_edges(n, [], []))
    rng = np.random.default_rng(n)
    for k in sorted({0, n // 10, n // 2, n}):
        pop = np.stack([rng.permutation(n)[:k] for _ in range(3)]).astype(np.int32)
        if k > 2:
            pop[1, 1] = pop[1, 0]  # a repeated gene counts once
        want = sx.fitness(g.row_ptr, g.col, pop, hops=hops, objective=objective)
        assert np.array_equal(_fit(ctx, g, pop, hops, objective, BITS), want), k


# the widest graph of four words per strip and the first of two, and the largest size, against the
# dense products
@pytest.mark.parametrize("n", [7000, 7300, 8192])
@pytest.mark.parametrize("objective", ["pc", "mcn"])
def test_bits_match_dense_products(ctx, n, objective):
    g = synth.hk_graph(n, 2, 0.3, 1)
    pop = synth.random_deletion_sets(n, n // 20, 3, 2)
    want = _fit(ctx, g, pop, 5, objective, TMA)
    assert np.array_equal(_fit(ctx, g, pop, 5, objective, BITS), want)
    assert np.array_equal(_fit(ctx, g, pop, 5, objective, AUTO), want)


# AUTO takes the dense products on a dense graph and bit rows on a sparse one
@pytest.mark.parametrize("edges,hops", [(20000, 9), (300, 9)])
def test_auto_route_matches_dense_reference(ctx, edges, hops):
    g = synth.er_graph(256, edges, 3)
    pop = synth.random_deletion_sets(256, 25, 20, 5)
    for objective in ("pc", "mcn"):
        want = sx.fitness(g.row_ptr, g.col, pop, hops=hops, objective=objective)
        assert np.array_equal(_fit(ctx, g, pop, hops, objective, AUTO), want)


def test_bits_report_bad_genes(ctx):
    import torch

    from paper_2412_20980_gb300 import GapaError

    g = synth.ba_graph(300, 2, 1)
    pop = synth.random_deletion_sets(300, 20, 4, 1)
    want = _fit(ctx, g, pop, 6, "pc", BITS)
    bad = pop.copy()
    bad[2, 5] = 300
    with pytest.raises(GapaError):
        _fit(ctx, g, bad, 6, "pc", BITS)
    assert np.array_equal(_fit(ctx, g, pop, 6, "pc", BITS), want)
