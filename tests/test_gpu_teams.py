"""Small teams of the sparse kernel and the (mu+lambda) ranks against the oracle at the edges of their rules."""
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


# rounds of members per SM on either side of 2, 4 and 6 teams, in one context as the scratch grows and shrinks
@pytest.mark.parametrize("n,k", [(37, 3), (400, 399), (1500, 75)])
@pytest.mark.parametrize("objective", ["pc", "mcn"])
def test_sparse_teams_match_oracle(ctx, n, k, objective):
    import torch

    from paper_2412_20980_gb300.gapa import FITNESS_SPARSE, OBJECTIVE_MCN, OBJECTIVE_PC

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = synth.ba_graph(n, 3, 1)
    rng = np.random.default_rng(n)
    ctx.graph_upload(g.row_ptr, g.col)
    ctx.set_fitness_kernel(FITNESS_SPARSE)
    ctx.set_objective(OBJECTIVE_MCN if objective == "mcn" else OBJECTIVE_PC)
    try:
        for s in (4 * sms - 1, 4 * sms, 8 * sms, 12 * sms - 1, 12 * sms, 5):
            pop = np.argsort(rng.random((s, n)), axis=1)[:, :k].astype(np.int32)
            pop[::3, 0] = 0  # a hub, maybe twice
            want = oracle.fitness(g.row_ptr, g.col, pop, "mcn" if objective == "mcn" else "bfs", nthreads=oracle.max_threads())
            got = ctx.fitness(torch.from_numpy(pop).cuda())
            ctx.sync()
            assert np.array_equal(got.cpu().numpy(), want), s
    finally:
        ctx.set_fitness_kernel(0)
        ctx.set_objective(OBJECTIVE_PC)


# entries per CTA and keys per round, one gene, more children than members and fewer, many equal keys
@pytest.mark.parametrize("mu,lam,k", [(2, 2, 1), (7, 2, 33), (5, 256, 3), (130, 131, 1), (64, 1030, 257)])
def test_mu_plus_lambda_ranks_match_oracle(ctx, mu, lam, k):
    from test_gpu_ga import MPL, _gen_case

    _gen_case(ctx, synth.ba_graph(300, 2, 1), k, mu, 0.6, 0.05, 2, 9, MPL, 3, lam=lam)
