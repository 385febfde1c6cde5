"""GPU parity of the greedy over candidate nodes: seeds and covered counts equal the oracle's
greedy on the same store where all nodes are candidates, where thousands of nodes tie around
the candidates' threshold (further epochs, the full index), where every set is covered before
the last seed, with sets of thousands of members, with no sets, and beside an open stepwise
selection."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
SID = O.make_sid(3, 0, 0)


def _run(g, w, model, theta, ks, seed=5):
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, model)
        tim.tim_sample_rr(eng.ctx, theta, seed, SID)
        off, mem, _ = tim.tim_get_rr(eng.ctx)
        counts = np.bincount(mem, minlength=g.n)
        assert np.array_equal(tim.tim_coverage_counts(eng.ctx, g.n), counts)
        rseeds, _, rcov = O.greedy(g.n, off, mem, max(ks))
        for k in ks:
            seeds, frac, cov = tim.tim_node_select(eng.ctx, k)
            assert np.array_equal(seeds, rseeds[:k])
            hit = np.isin(mem, seeds)
            assert cov == np.unique(np.repeat(np.arange(theta), np.diff(off))[hit]).size
            assert frac == (cov / theta if theta else 0.0)


@pytest.mark.parametrize("theta", [0, 1, 3, 4000, 60_000])
def test_skewed_store(theta):
    g = inputs.rmat(14, seed=41)
    _run(g, inputs.weighted_cascade(g), O.IC, theta, (1, 50, 400))


@pytest.mark.parametrize("n,theta", [(30_000, 20_000), (200_000, 50_000)])
def test_ties_around_the_threshold(n, theta):
    # every set is its root alone: thousands of nodes with the same small counts
    g = inputs.from_edges(n, [(0, 1)])
    _run(g, inputs.constant(g, 0.0), O.IC, theta, (1, 40, 3000))


def test_everything_covered_early():
    g = inputs.star_in(3000)  # node 0 reaches itself only; every other set holds its root
    _run(g, inputs.constant(g, 1.0), O.IC, 500, (1, 450, 2999))
    g = inputs.cycle(50)  # p = 1: every set holds every node
    _run(g, inputs.constant(g, 1.0), O.IC, 300, (1, 2, 50))


@pytest.mark.parametrize("n,m,theta", [(1500, 3600, 400), (12_000, 30_000, 150),
                                       (60_000, 240_000, 40)])
def test_large_sets(n, m, theta):
    # p = 1: sets of about a thousand, thousands and more than 32,768 members, shared by a
    # block's warps or by all of them
    g = inputs.random_small(n, m, seed=3)
    _run(g, inputs.constant(g, 1.0), O.IC, theta, (1, 30))


def test_uniform_store_many_seeds():
    g = inputs.random_small(20_000, 40_000, seed=7)
    _run(g, inputs.lt_inverse_indegree(g), O.LT, 30_000, (5, 1500))


def test_beside_an_open_stepwise_selection():
    g = inputs.rmat(12, seed=42)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, inputs.weighted_cascade(g), O.IC)
        tim.tim_sample_rr(eng.ctx, 5000, 5, SID)
        off, mem, _ = tim.tim_get_rr(eng.ctx)
        rseeds, rcov, _ = O.greedy(g.n, off, mem, 8)
        tim.tim_select_begin(eng.ctx)
        first = tim.tim_select_take(eng.ctx, int(rseeds[0]))
        assert first == np.bincount(mem, minlength=g.n)[rseeds[0]]
        seeds, _, cov = tim.tim_node_select(eng.ctx, 8)
        assert np.array_equal(seeds, rseeds)
        # the stepwise calls go on from the sets that selection left uncovered
        left = tim.tim_select_counts(eng.ctx, g.n)
        hit = np.zeros(len(off) - 1, dtype=bool)
        sid = np.repeat(np.arange(len(off) - 1), np.diff(off))
        hit[sid[np.isin(mem, rseeds)]] = True
        assert cov == hit.sum()
        assert np.array_equal(left, np.bincount(mem[~hit[sid]], minlength=g.n))


@pytest.mark.parametrize("n,theta,ks", [
    (30_000, 150_000, (3, 5, 6)), (30_000, 150_001, (3, 5, 6)),  # the largest small store
    (2_000_000, 12_000, (5, 6, 30, 45, 127, 128, 129, 300))])  # some 36 nodes in two sets
def test_few_seeds_and_few_candidates(n, theta, ks):
    # every set is its root alone
    g = inputs.from_edges(n, [(0, 1)])
    _run(g, inputs.constant(g, 0.0), O.IC, theta, ks)
