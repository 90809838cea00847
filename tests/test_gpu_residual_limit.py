"""Residual counts of the largest graph whose deletion bitmap fits in shared memory."""
import numpy as np
import pytest

import synth
from test_gpu_residual import _counts

pytestmark = pytest.mark.gpu


def test_residual_counts_at_the_size_limit():
    import torch

    from paper_2412_20980_gb300 import Context, GapaError, Surrogate, make_surrogate_config

    # 227 KB less the kernel's 96 static bytes, eight nodes per byte
    n = 8 * (torch.cuda.get_device_properties(0).shared_memory_per_block_optin - 96)
    rng = np.random.default_rng(n)
    u, v = rng.integers(0, n, (2, n // 2))
    hub = rng.integers(1, n, 5000)  # a long adjacency beside the short ones
    u, v = np.concatenate([u, np.zeros_like(hub)]), np.concatenate([v, hub])
    g = synth.csr_from_edges(n, u[u != v], v[u != v])
    pop = np.stack([rng.permutation(n)[:3000] for _ in range(3)]).astype(np.int32)
    pop[1, 0] = 0
    pop[2, 1] = pop[2, 0]
    with Context(0) as ctx:
        ctx.graph_upload(g.row_ptr, g.col)
        sg = Surrogate(ctx, make_surrogate_config(batch=16, ring=16), seed=1)
        got = sg.residual(torch.from_numpy(pop).cuda()).cpu().numpy()
        assert np.array_equal(got, _counts(g, pop))
        sg.close()
        big = synth.csr_from_edges(n + 1, [0], [n])
        ctx.graph_upload(big.row_ptr, big.col)
        with pytest.raises(GapaError):
            Surrogate(ctx, make_surrogate_config(batch=16, ring=16), seed=1)
