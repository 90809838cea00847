"""The cut-local kernel's shared-memory layout up to the largest graph that it takes, and the graphs on which
the automatic setting takes it.

The launch shape is plain C++: a host program walks every graph size, and the sizes next to the limits
run on the GPU against the oracle.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_20980_gb300", "csrc")

CHECK = r"""
#include "local_layout.cuh"
using namespace gapa_dev;
// First n up to `top` whose launch breaks a rule (0: none); *rule says which.
extern "C" int check(int top, int deg16, int s, int sms, size_t per_sm, size_t reserved, size_t block_max, int* rule) {
    const LocalLimits d{sms, per_sm, reserved, block_max};
    for (int n = 1; n <= top; ++n) {
        if (!local_admits(n, deg16, block_max)) continue;
        const LocalShape x = local_shape(n, deg16, s, d);
        const size_t list = (size_t)x.list_bytes, smem = tree16l_smem_bytes(n, list);
        *rule = x.list_bytes <= 0 || list % 16 ? 1                    // whole 16-byte units
              : list < tree16l_min_list_bytes(n, deg16) ? 2           // what the fallbacks need
              : smem > block_max ? 3                                  // within the block's limit
              : x.per_sm > 1 && x.per_sm * (smem + reserved) > per_sm ? 4
              : x.threads % 32 || x.threads < 32 || x.threads > 1024 || x.threads * x.per_sm > 2048 ? 5
              // the fallbacks' own extents: bitmap and four scalars, or 32-bit labels, bitmap and scalars
              : (size_t)((n + 31) / 32) * 4 + 16 > list ? 6
              : tree16l_tops_max(n, deg16) < n && tree32_smem_bytes(n) > tree16_lab_bytes(n) + list ? 7 : 0;
        if (*rule) return n;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    (d / "check.cpp").write_text(CHECK)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "check.cpp"), "-o",
                    str(d / "check.so")], check=True)
    lib = ctypes.CDLL(str(d / "check.so"))
    size = ctypes.c_size_t
    lib.check.argtypes = [ctypes.c_int] * 4 + [size] * 3 + [ctypes.POINTER(ctypes.c_int)]
    return lib


# both sides of a mean degree of 5, one to eight members per SM; a block's limit is 227 KB less the
# kernels' static shared memory (272 bytes, and round values about it)
@pytest.mark.parametrize("deg16", [16, 47, 64, 79, 80, 160])
@pytest.mark.parametrize("static", [0, 272, 640, 1024])
def test_layout_holds_every_fallback(layout, deg16, static):
    sms, per_sm, reserved, optin = 152, 228 * 1024, 1024, 227 * 1024
    for s in (1, sms, sms + 1, 2 * sms + 1, 3 * sms + 1, 4 * sms + 1, 5 * sms + 1, 6 * sms + 1, 7 * sms + 1, 10000):
        rule = ctypes.c_int(0)
        n = layout.check(65534, deg16, s, sms, per_sm, reserved, optin - static, ctypes.byref(rule))
        assert n == 0, f"n = {n}, s = {s}: rule {rule.value}"


# sets of more than n / 5 tops, which a graph of two links per node hands to the 32-bit pipeline, at the
# largest sizes of the kernel and past them
@pytest.mark.gpu
@pytest.mark.parametrize("n", [56083, 56084, 56099, 56265, 56284])
def test_largest_graphs_match_oracle(layout, n):
    import torch

    from paper_2412_20980_gb300 import Context, build
    from paper_2412_20980_gb300.gapa import FITNESS_PIECE, FITNESS_TREE_LOCAL, OBJECTIVE_MCN, OBJECTIVE_PC

    build.build()
    g = synth.ba_graph(n, 2, 1)
    rng = np.random.default_rng(n)
    order = np.argsort(-g.degrees(), kind="stable").astype(np.int32)
    k, s = n // 6, 160
    pop = np.stack([rng.permutation(n)[:k] for _ in range(s)]).astype(np.int32)
    for i in range(0, s, 2):  # half of the genes among the hubs, so more tops than n / 5
        rest = order[k // 2:]
        pop[i] = np.concatenate([order[:k // 2], rest[rng.permutation(rest.size)[:k - k // 2]]])
    pop[3, 1] = pop[3, 0]  # a repeated gene: the 16-bit pipeline
    with Context(0) as ctx:
        ctx.graph_upload(g.row_ptr, g.col)
        for name, objective in (("bfs", OBJECTIVE_PC), ("mcn", OBJECTIVE_MCN)):
            want = oracle.fitness(g.row_ptr, g.col, pop, name, nthreads=oracle.max_threads())
            ctx.set_objective(objective)
            for kernel in (0, FITNESS_TREE_LOCAL, FITNESS_PIECE):
                ctx.set_fitness_kernel(kernel)
                got = ctx.fitness(torch.from_numpy(pop).cuda())
                ctx.sync()
                assert np.array_equal(got.cpu().numpy(), want), (name, kernel)


# by the launches of a call that does not fit the SMs at once: the full pipeline is one, the cut-local kernel
# comes after its cost estimates and order
@pytest.mark.gpu
@pytest.mark.parametrize("n,edges,launches", [(649, "ba", 1), (650, "ba", 3), (300, 1800, 1), (950, 2849, 1), (1000, 2850, 3), (500, 2850, 3),
                                              (2000, 5600, 1), (2048, 5888, 3), (2049, 3074, 3), (2049, 3009, 1)])
def test_automatic_choice_on_both_sides_of_its_lines(n, edges, launches):
    import torch

    from paper_2412_20980_gb300 import Context, build

    build.build()
    g = synth.ba_graph(n, 4, 1) if edges == "ba" else synth.er_graph(n, edges, 7)
    s = 9 * torch.cuda.get_device_properties(0).multi_processor_count
    pop = synth.random_deletion_sets(n, n // 20, s, 5)
    with Context(0) as ctx:
        ctx.graph_upload(g.row_ptr, g.col)
        dev = torch.from_numpy(pop).cuda()
        ctx.profile_begin()
        got = ctx.fitness(dev)
        ctx.sync()
        assert ctx.profile_end()["fitness_launches"] == launches
        assert np.array_equal(got.cpu().numpy(), oracle.fitness(g.row_ptr, g.col, pop, nthreads=oracle.max_threads()))
