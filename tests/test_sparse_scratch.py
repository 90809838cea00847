"""The sparse kernel's scratch: how it grows with the population, and what it holds between members."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_20980_gb300", "csrc")

GROW = r"""
#include "sparse_layout.cuh"
using namespace gapa_dev;
// The shape held after asking for `shape`; room: the shapes below it fit in the device; *asked: allocations.
extern "C" int grow(int held, int shape, int may_grow, int* refused, int room, int* asked) {
    return sp_grow(held, shape, may_grow != 0, refused, [&](int i) { ++*asked; return i < room; });
}
extern "C" int shape(int n, int deg16, int s, int k) { return sp_shape(n, deg16, s, k, SpLimits{152, 228 * 1024, 1024}); }
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("scratch")
    (d / "grow.cpp").write_text(GROW)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "grow.cpp"), "-o",
                    str(d / "grow.so")], check=True)
    return ctypes.CDLL(str(d / "grow.so"))


@pytest.mark.parametrize("room", range(4))
@pytest.mark.parametrize("held,shape", [(-1, 0), (-1, 2), (0, 2), (0, 1), (2, 1), (1, 2)])
def test_growth_steps_down_and_asks_once(layout, room, held, shape):
    refused, asked = ctypes.c_int(3), ctypes.c_int(0)
    call = lambda h, s, may=1: layout.grow(h, s, may, ctypes.byref(refused), room, ctypes.byref(asked))
    want = max(held, min(shape, room - 1))
    assert call(held, shape) == want  # the largest that there is room for, and none given up
    if 0 <= want < shape:  # a shape refused is not asked for again
        seen = asked.value
        assert call(want, shape) == want and asked.value == seen


def test_no_growth_inside_a_capture(layout):
    refused, asked = ctypes.c_int(3), ctypes.c_int(0)
    assert layout.grow(0, 2, 0, ctypes.byref(refused), 3, ctypes.byref(asked)) == 0
    assert asked.value == 0 and refused.value == 3


# what small teams were measured slower on keeps one member per SM: trees and graphs of mean degree 3, less
# than eight members per SM, more nodes than the slices' reads stay in L2 for
@pytest.mark.parametrize("n,deg16,s,k,want", [
    (60000, 32, 4096, 200, 0), (200000, 48, 4096, 2000, 0), (60000, 56, 1216, 200, 1),
    (100000, 96, 1215, 2000, 0), (100000, 96, 1216, 2000, 1), (100000, 96, 1823, 2000, 1), (100000, 96, 1824, 2000, 2),
    (109649, 96, 2048, 2000, 2), (109650, 96, 2048, 2000, 1), (263157, 128, 4096, 2000, 1),
    (263158, 128, 4096, 2000, 0), (1 << 20, 128, 4096, 200, 0)])
def test_small_teams_where_they_gain(layout, n, deg16, s, k, want):
    assert layout.shape(n, deg16, s, k) == want


# the shapes that the device chooses between, by the launches of a call (cost, order, and one kernel or both)
@pytest.mark.gpu
@pytest.mark.parametrize("graph,per_sm,launches", [("ba", 8, 4), ("ba", 12, 4), ("tree", 12, 3)])
def test_shapes_on_both_sides_of_a_rule_match_oracle(ctx, graph, per_sm, launches):
    import torch

    n, sms = 1500, torch.cuda.get_device_properties(0).multi_processor_count
    g = synth.ba_graph(n, 3 if graph == "ba" else 1, 1)
    ctx.graph_upload(g.row_ptr, g.col)
    order = np.argsort(-g.degrees(), kind="stable").astype(np.int32)
    for s, want in ((per_sm * sms - 1, 3 if per_sm == 8 else launches), (per_sm * sms, launches)):
        for hubs in (False, True):  # light members alike, heavy ones
            pop = synth.random_deletion_sets(n, 75, s, s)
            if hubs:
                pop[:, :40] = order[:40]
            ctx.profile_begin()
            got = _fitness(ctx, pop)
            assert ctx.profile_end()["fitness_launches"] == want
            assert np.array_equal(got, oracle.fitness(g.row_ptr, g.col, pop, nthreads=oracle.max_threads())), (s, hubs)


@pytest.fixture(scope="module")
def ctx():
    from paper_2412_20980_gb300 import Context
    from paper_2412_20980_gb300 import build as b
    from paper_2412_20980_gb300.gapa import FITNESS_SPARSE

    b.build()
    with Context(0) as c:
        c.set_fitness_kernel(FITNESS_SPARSE)
        yield c


def _fitness(ctx, pop):
    import torch

    out = ctx.fitness(torch.from_numpy(pop).cuda())
    ctx.sync()
    return out.cpu().numpy()


# a call with more members than any before it on this graph, captured: the blocks held serve
@pytest.mark.gpu
def test_captured_call_of_a_larger_population():
    import torch

    from paper_2412_20980_gb300 import Context
    from paper_2412_20980_gb300.gapa import FITNESS_SPARSE

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), Context(0) as c:
        c.set_fitness_kernel(FITNESS_SPARSE)
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        for n, s in ((1000, 14 * sms), (3000, 5)):  # the member order is sized by the first, the slices by the second
            g = synth.ba_graph(n, 3, 1)
            c.graph_upload(g.row_ptr, g.col)
            pop = synth.random_deletion_sets(n, n // 20, s, 3)
            assert np.array_equal(_fitness(c, pop), oracle.fitness(g.row_ptr, g.col, pop, nthreads=oracle.max_threads()))
        pop = synth.random_deletion_sets(n, n // 20, 14 * sms, 4)
        dev, out = torch.from_numpy(pop).cuda(), torch.zeros(14 * sms, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            c.fitness(dev, out)
        graph.replay()
        torch.cuda.synchronize()
        want = oracle.fitness(g.row_ptr, g.col, pop, nthreads=oracle.max_threads())
        assert np.array_equal(out.cpu().numpy(), want)
        assert np.array_equal(_fitness(c, pop), want)  # outside it the blocks grow
        out.zero_()
        graph.replay()  # and those that the capture holds are still there
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)


# graphs of one stride after one another in one context, connected ones and ones of many components and
# single nodes, their numbers of members on both sides of every shape: nothing of one member or graph is
# left for the next
@pytest.mark.gpu
@pytest.mark.parametrize("objective", ["pc", "mcn"])
def test_members_and_graphs_leave_nothing_behind(ctx, objective):
    import torch

    from paper_2412_20980_gb300.gapa import OBJECTIVE_MCN, OBJECTIVE_PC

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 1990
    rng = np.random.default_rng(3)
    u, v = rng.integers(0, n, (2, int(1.1 * n)))
    back = (np.arange(1, n) * rng.random(n - 1)).astype(np.int64)
    graphs = [synth.ba_graph(n, 3, 1), synth.csr_from_edges(n, u[u != v], v[u != v]),
              synth.csr_from_edges(n, back, np.arange(1, n)),
              synth.graphs.disjoint_union(synth.hk_graph(990, 4, 0.3, 1), synth.named_graph("star", 500),
                                          synth.named_graph("empty", 100), synth.ba_graph(400, 2, 2))]
    ctx.set_objective(OBJECTIVE_MCN if objective == "mcn" else OBJECTIVE_PC)
    try:
        for s in (sms, 13 * sms, 3, 8 * sms):
            for g in graphs:
                ctx.graph_upload(g.row_ptr, g.col)
                order = np.argsort(-g.degrees(), kind="stable").astype(np.int32)
                k = 150
                pop = synth.random_deletion_sets(n, k, s, s)
                pop[::2, :k // 3] = order[:k // 3]  # hubs, some of them twice
                want = oracle.fitness(g.row_ptr, g.col, pop, "mcn" if objective == "mcn" else "bfs",
                                      nthreads=oracle.max_threads())
                assert np.array_equal(_fitness(ctx, pop), want), s
    finally:
        ctx.set_objective(OBJECTIVE_PC)
