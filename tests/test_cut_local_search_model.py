"""The cut-local kernel's steps on the CPU, every access to the shared 16-bit labels in a random
interleaving, against the oracle.

Per member (tree16_local_try): the children of deleted nodes ("tops") take a live lower-numbered
neighbour as label, those without one ("terminals") are united with up to two live higher-numbered
neighbours; R is the first live node or, where node 0 is deleted, the root that most of a few live
nodes reach, so it need not be the smallest of its class; the terminals and component roots that are
still roots and not R seed a list, from which a breadth-first search over live arcs runs: a neighbour
in R's class joins the node's class to R, any other is united with it and listed.  What is not listed
lies in R's class.

Two labels share a 32-bit word: a union swaps one of them by a compare-and-swap of the word, path
halving and a newly listed child store one half.  A node hooks under a smaller root, or under R
whatever R's number; a store goes to a node that is no root and names an ancestor.
"""
import random

import numpy as np
import pytest

import oracle
import synth
from synth.graphs import disjoint_union
from test_concurrency_models import run_interleaved
from test_cut_local_model import bfs_numbering, children_runs

DEAD = 0xFFFF


class Labels:
    """Labels two to a word; every method yields before each access to a word."""

    def __init__(self, values):
        values = list(values) + [0] * (len(values) % 2)
        self.w = [values[i] | values[i + 1] << 16 for i in range(0, len(values), 2)]

    def now(self, i):
        return self.w[i >> 1] >> (16 * (i & 1)) & 0xFFFF

    def put(self, i, v):
        sh = 16 * (i & 1)
        self.w[i >> 1] = self.w[i >> 1] & ~(0xFFFF << sh) | v << sh

    def load(self, i):
        yield
        return self.now(i)

    def store(self, i, v):
        yield
        self.put(i, v)

    def cas(self, i, expect, v):
        sh = 16 * (i & 1)
        yield
        old = self.w[i >> 1]
        while True:
            cur = old >> sh & 0xFFFF
            if cur != expect:
                return cur
            yield
            seen = self.w[i >> 1]
            if seen == old:
                self.w[i >> 1] = old & ~(0xFFFF << sh) | v << sh
                return cur
            old = seen


def find(lab, x):
    while True:
        p = yield from lab.load(x)
        if p == x:
            return x
        gp = yield from lab.load(p)
        if gp == p:
            return p
        yield from lab.store(x, gp)
        x = gp


def unite(lab, a, b, R=-1):
    a = yield from find(lab, a)
    b = yield from find(lab, b)
    while a != b:
        if b != R and (a == R or a < b):
            a, b = b, a
        old = yield from lab.cas(a, a, b)
        if old == a:
            return
        a = yield from find(lab, old)
        b = yield from find(lab, b)


def root(lab, x):
    while lab.now(x) != x:
        assert lab.now(x) != DEAD
        x = lab.now(x)
    return x


def member(tparent, adj, kids, singles, dead, rng, vote, lanes=4):
    """(PC, MCN, listed) of one member; vote(live nodes' roots) picks R where node 0 is deleted."""
    n = len(tparent)
    lab = Labels([DEAD if x in dead else tparent[x] for x in range(n)])
    live = [x for x in range(n) if x not in dead]
    others = [x for x in live if x not in singles]
    if not others:
        return 0, int(bool(live)), set()
    terms = []
    for c in (c for d in dead for c in kids[d] if c not in dead):
        lower = [w for w in adj[c] if w < c][1:]  # the second to fourth and the last
        pick = [w for w in lower[:3] + lower[-1:] if w not in dead]
        lab.put(c, pick[0] if pick else c)
        if not pick:
            terms.append(c)

    def link(c):
        higher = sorted((w for w in adj[c] if w > c and tparent[w] != c), key=lambda w: -len(adj[w]))[:4]
        for w in [w for w in higher if w not in dead][:2]:
            yield from unite(lab, c, w)

    run_interleaved([link(c) for c in terms], rng)
    R = live[0] if live[0] == 0 else vote([root(lab, x) for x in live])
    assert lab.now(R) == R
    seeds = [c for c in terms if c != R and lab.now(c) == c]
    seeds += [x for x in range(n) if tparent[x] == x and adj[x] and x not in dead and x != R and lab.now(x) == x]
    found, marked = list(seeds), set(seeds)

    def arcs(v, sub):
        at_r = yield from find(lab, v)
        if at_r == R:
            return
        for w in adj[v][sub::lanes]:
            lw = yield from lab.load(w)
            if lw == DEAD:
                continue
            below = lw == v
            if w not in marked:
                if not below and (yield from find(lab, w)) == R:
                    yield from unite(lab, v, R, R)
                    return
                yield
                if w not in marked:  # one atomic operation
                    marked.add(w)
                    found.append(w)
                    if below:
                        up = yield from lab.load(v)
                        yield from lab.store(w, up)
            if not below:
                a = yield from lab.load(w)
                b = yield from lab.load(v)
                if a != b:
                    yield from unite(lab, v, w, R)

    head = 0
    while head < len(found):
        tail = len(found)
        run_interleaved([arcs(v, sub) for v in found[head:tail] for sub in range(lanes)], rng)
        head = tail
    sizes = {}
    for x in found:
        sizes[root(lab, x)] = sizes.get(root(lab, x), 0) + 1
    joined = sizes.pop(R, 0)
    sizes[R] = len(others) - len(found) + joined
    mcn = max(max(sizes.values()), int(any(x in singles for x in live)))
    return sum(c * (c - 1) // 2 for c in sizes.values()), mcn, set(found)


GRAPHS = {
    "ba": lambda: synth.ba_graph(120, 2, 1),
    "hk": lambda: synth.hk_graph(120, 3, 0.3, 2),
    "er_sparse": lambda: synth.er_graph(140, 150, 3),  # many components and single nodes
    "union": lambda: disjoint_union(synth.ba_graph(70, 2, 4), synth.named_graph("path", 30),
                                    synth.named_graph("star", 20), synth.named_graph("empty", 6)),
}


# R by majority, as the kernel does, and any root at all: the choice never shows in the result
@pytest.mark.parametrize("choice", ["majority", "any"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_interleaved_members_match_oracle(name, choice):
    g = GRAPHS[name]()
    num, tparent, adj = bfs_numbering(g)
    kids = children_runs(tparent)
    singles = {x for x in range(g.n) if not adj[x]}
    top = np.argsort(-g.degrees(), kind="stable")
    rng = np.random.default_rng(len(name))
    k = g.n // 8
    rows = [rng.choice(g.n, k, replace=False) for _ in range(4)]
    rows += [np.concatenate([top[:h], rng.choice(top[h:], k - h, replace=False)]) for h in (1, 3, k // 2, k)]
    pop = np.stack(rows).astype(np.int32)
    want_pc, want_mcn = oracle.fitness(g.row_ptr, g.col, pop), oracle.fitness(g.row_ptr, g.col, pop, "mcn")
    for i, row in enumerate(pop):
        sched = random.Random(31 * i + len(choice))
        vote = (lambda roots: max(set(roots), key=roots.count)) if choice == "majority" else sched.choice
        pc, mcn, listed = member(tparent, adj, kids, singles, {num[int(d)] for d in row}, sched, vote)
        assert (pc, mcn) == (want_pc[i], want_mcn[i]), (i, listed)


def test_edge_members():
    g = GRAPHS["union"]()
    num, tparent, adj = bfs_numbering(g)
    kids = children_runs(tparent)
    singles = {x for x in range(g.n) if not adj[x]}
    majority = lambda roots: max(set(roots), key=roots.count)
    run = lambda dead: member(tparent, adj, kids, singles, dead, random.Random(1), majority)[:2]
    assert run(set(range(g.n))) == (0, 0)  # nothing left
    assert run(set(range(g.n)) - singles) == (0, 1)  # single nodes alone
    ids = {int(num[v]): v for v in range(g.n)}
    for dead in (set(), {0}, {0} | set(kids[0]), set(kids[0])):
        pop = np.array([[ids[x] for x in sorted(dead)]], dtype=np.int32)
        assert run(dead) == (oracle.fitness(g.row_ptr, g.col, pop)[0], oracle.fitness(g.row_ptr, g.col, pop, "mcn")[0])


@pytest.mark.parametrize("seed", range(20))
def test_unions_towards_any_root(seed):
    """Unions under random schedules with R anywhere: the classes are those of the edges, R stays a root,
    and every label's walk ends (a store that named no ancestor, or a root hooked under two, would not)."""
    rng = random.Random(seed)
    n = rng.choice([9, 24, 41])
    lab = Labels(range(n))
    R = rng.randrange(n)
    edges = [(rng.randrange(n), rng.randrange(n)) for _ in range(2 * n // 3)]
    run_interleaved([unite(lab, a, b, R) for a, b in edges], rng)
    assert lab.now(R) == R
    part = list(range(n))
    for _ in range(n):
        for a, b in edges:
            part[a] = part[b] = min(part[a], part[b])
    roots = [root(lab, x) for x in range(n)]
    assert all((roots[a] == roots[b]) == (part[a] == part[b]) for a in range(n) for b in range(n))
