"""The forest-piece kernel's tables come with the choice of that kernel, before or after the graph's upload."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chosen", ["before", "after", "before a second graph"])
def test_tables_are_there_when_the_kernel_runs(chosen):
    import torch

    from paper_2412_20980_gb300 import Context, build
    from paper_2412_20980_gb300.gapa import FITNESS_PIECE

    build.build()
    g = synth.ba_graph(3000, 3, 4)
    pop = synth.random_deletion_sets(g.n, 150, 40, 2)
    with Context(0) as ctx:
        if chosen != "after":
            ctx.set_fitness_kernel(FITNESS_PIECE)
        if chosen == "before a second graph":
            other = synth.ba_graph(700, 2, 1)
            ctx.graph_upload(other.row_ptr, other.col)
        ctx.graph_upload(g.row_ptr, g.col)
        if chosen == "after":
            ctx.set_fitness_kernel(FITNESS_PIECE)
        dev = torch.from_numpy(pop).cuda()
        ctx.profile_begin()
        got = ctx.fitness(dev)
        ctx.sync()
        # the full pipeline, which serves without the tables, is one launch
        assert ctx.profile_end()["fitness_launches"] > 3
        assert np.array_equal(got.cpu().numpy(), oracle.fitness(g.row_ptr, g.col, pop, nthreads=oracle.max_threads()))
