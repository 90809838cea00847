"""Residual counts where the choice of kernel changes: the largest graph whose deletion bitmap fits in shared
memory, and few or many genes and rows on graphs with long and with short adjacencies."""
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


# with the once / twice bitmaps and without (few genes on graphs of short adjacencies, many rows), 256 to 1024
# threads per row
@pytest.mark.parametrize("n,rows,k", [(30000, 1300, 20), (30000, 1300, 700), (160000, 330, 40), (160000, 330, 1100),
                                      (160000, 150, 40), (420000, 310, 600)])
@pytest.mark.parametrize("shape", ["even", "hubs"])
def test_residual_counts_by_either_kernel(n, rows, k, shape):
    import torch

    from paper_2412_20980_gb300 import Context, Surrogate, make_surrogate_config

    rng = np.random.default_rng(n + k)
    u, v = rng.integers(0, n, (2, int(1.6 * n)))
    if shape == "hubs":
        v[: n // 4] = rng.integers(0, 30, n // 4)
    g = synth.csr_from_edges(n, u[u != v], v[u != v])
    pop = np.stack([rng.permutation(n)[:k] for _ in range(8)]).astype(np.int32)
    pop[::2, :8] = np.argsort(-np.diff(g.row_ptr), kind="stable")[:8]  # the longest adjacencies, some genes twice
    pop[0, :2] = (-1, n)  # ignored
    full = np.concatenate([pop] * (rows // 8 + 1))[:rows]
    with Context(0) as ctx:
        ctx.graph_upload(g.row_ptr, g.col)
        sg = Surrogate(ctx, make_surrogate_config(batch=16, ring=16), seed=1)
        got = sg.residual(torch.from_numpy(full).cuda()).cpu().numpy()
        want = _counts(g, pop)
        assert np.array_equal(got, np.concatenate([want] * (rows // 8 + 1))[:rows])
        sg.close()
