"""The automatic SixDST setting takes bit rows where they cost less and the dense products elsewhere, by the
launches of a call: bit rows are one, the products several."""
import numpy as np
import pytest

import synth
from oracle import sixdst_ref as sx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edges,bits", [(20000, False), (300, True)])
@pytest.mark.parametrize("objective", ["pc", "mcn"])
def test_route_and_result(edges, bits, objective):
    import torch

    from paper_2412_20980_gb300 import Context, build
    from paper_2412_20980_gb300.gapa import OBJECTIVE_SIXDST_MCN, OBJECTIVE_SIXDST_PC

    build.build()
    g = synth.er_graph(256, edges, 3)
    pop = synth.random_deletion_sets(256, 25, 20, 5)
    with Context(0) as ctx:
        ctx.graph_upload(g.row_ptr, g.col)
        ctx.set_objective(OBJECTIVE_SIXDST_MCN if objective == "mcn" else OBJECTIVE_SIXDST_PC)
        ctx.set_sixdst_hops(9)
        dev = torch.from_numpy(pop).cuda()
        ctx.profile_begin()
        got = ctx.fitness(dev)
        ctx.sync()
        launches = ctx.profile_end()["fitness_launches"]
        assert (launches == 1) if bits else (launches > 3)
        assert np.array_equal(got.cpu().numpy(), sx.fitness(g.row_ptr, g.col, pop, hops=9, objective=objective))
