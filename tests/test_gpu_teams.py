"""Small teams of the sparse kernel, the (mu+lambda) ranks and packed batch results against the oracle at the edges of their rules."""
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


# one object over longer and shorter runs and other teams: results, trajectories and sets of every size
@pytest.mark.parametrize("ks", [(0, 1, 31, 2000), (2999, 0, 0, 1)])
def test_batch_results_of_repeated_runs_match_oracle(ks):
    from paper_2412_20980_gb300 import Batch, Context, make_config

    graphs = [synth.ba_graph(n, 3, 5) for n in (3000, 33, 64, 20011)]
    ctxs, cfgs = [], []
    for g, k in zip(graphs, ks):
        ctxs.append(Context(0))
        ctxs[-1].graph_upload(g.row_ptr, g.col)
        cfgs.append(make_config(k=k, pop=6, tourn=2, pc=0.8, pm=0.1, seed=k))
    bt = Batch(ctxs, cfgs)
    for gens, teams in [(2, None), (5, None), (0, None), (4, [2, 8, 4, 1]), (4, [1, 1, 1, 1])]:
        if teams:
            bt.teams = teams
        got = bt.run(gens)
        for i, (g, cfg) in enumerate(zip(graphs, cfgs)):
            want = oracle.run(g.row_ptr, g.col, k=cfg.k, pop=cfg.pop, gens=gens, tourn=cfg.tourn, pc_thr=cfg.pc_thr,
                              pm_thr=cfg.pm_thr, seed=cfg.seed, nthreads=oracle.max_threads())
            assert np.array_equal(got["traj"][i], want["traj"]), (gens, i)
            assert got["best_fit"][i] == want["best_fit"], (gens, i)
            assert np.array_equal(got["best_sets"][i], want["best_set"]), (gens, i)
    bt.close()
