"""GPU parity of Algorithm 2 when several of its rounds are sampled in one call, and of sets
that pass 2 hands to the heavy-set pass for their long in-lists: KPT*, stopping round and the
stopping (or last) round's RR sets in the store equal the oracle's, whichever rounds shared a
call -- stops at the first, second and later rounds, no stop at all, sets of every pass, IC,
LT and triggering models."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu


def _graph(name):
    if name == "wc":
        g = inputs.rmat(13, seed=21)
        return g, inputs.weighted_cascade(g), O.IC
    if name == "lt":
        g = inputs.rmat(13, seed=22)
        return g, inputs.lt_random_normalised(g, 2), O.LT
    if name == "triv":  # in-lists of thousands of in-edges, each with its own coin
        g = inputs.chung_lu(20_001, 500_000, 2.1, seed=23)
        return g, inputs.trivalency(g, seed=4), O.IC
    if name == "sparse":  # most roots have no in-edges: many rounds
        g = inputs.random_small(6000, 500, seed=24)
        return g, inputs.constant(g, 0.5), O.IC
    if name == "edge_free":  # no round stops: the last round's sets stay in the store
        g = inputs.from_edges(70, [])
        return g, inputs.constant(g, 1.0), O.IC
    if name == "p1":  # stops at once
        g = inputs.random_small(400, 3000, seed=25)
        return g, inputs.constant(g, 1.0), O.IC
    raise KeyError(name)


def _sorted_sets(off, mem):
    return [np.sort(mem[off[j]:off[j + 1]]).tolist() for j in range(len(off) - 1)]


def _check_kpt(eng, og, k, seed):
    ref = O.kpt_estimation(og, k, 1.0, seed)
    kpt, rnd = tim.tim_kpt_estimate(eng.ctx, k, 1.0, seed)
    assert rnd == ref.stop_round and kpt == ref.kpt_star
    last = rnd if rnd else O.kpt_rounds(og.n)
    off, mem, wid = tim.tim_get_rr(eng.ctx)
    c = O.c_i(og.n, 1.0, last)
    roff, rmem, rwid = O.sample(og, seed, O.make_sid(1, last, 0), c)
    assert np.array_equal(off, roff) and np.array_equal(wid, rwid)
    assert _sorted_sets(off, mem) == _sorted_sets(roff, rmem)
    return rnd


@pytest.mark.parametrize("name", ["wc", "lt", "triv", "sparse", "edge_free", "p1"])
def test_rounds_in_one_call(name):
    g, w, model = _graph(name)
    og = O.load_graph(g.n, g.rowptr, g.dst, w, model)
    stops = set()
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, model)
        for k, seed in ((1, 3), (2, 4), (10, 5), (40, 6)):
            stops.add(_check_kpt(eng, og, k, seed))
        # Algorithm 3 runs on the kept sets
        ref = O.refine_kpt(og, 10, 1.0, 0.5, 5, O.kpt_estimation(og, 10, 1.0, 5))
        tim.tim_kpt_estimate(eng.ctx, 10, 1.0, 5)
        kpt_plus, _, theta_prime = tim.tim_refine_kpt(eng.ctx, 10, 1.0, 0.5, 5)
        assert theta_prime == ref.theta_prime
        assert abs(kpt_plus - ref.kpt_plus) <= 1e-9 * ref.kpt_plus
    if name == "edge_free":
        assert stops == {0}
    if name == "p1":
        assert 1 in stops


def test_rounds_in_one_call_triggering():
    g = inputs.rmat(12, seed=31)
    opts = inputs.triggering_random(g, seed=6)
    og = O.load_graph_triggering(g.n, g.rowptr, g.dst, *opts)
    with tim.Engine(0) as eng:
        tim.tim_load_graph_triggering(eng.ctx, g.n, g.rowptr, g.dst, *opts)
        for k, seed in ((1, 3), (20, 4)):
            _check_kpt(eng, og, k, seed)


def test_long_lists_move_to_the_heavy_pass():
    g, w, model = _graph("triv")
    og = O.load_graph(g.n, g.rowptr, g.dst, w, model)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, model)
        sid, count = O.make_sid(3, 0, 0), 30_000
        for budget in (16384, 0):  # from pass 1's hand-over, and with every set in pass 2
            tim.tim_set_width_budget(eng.ctx, budget)
            tim.tim_get_profile(eng.ctx, reset=True)
            tim.tim_sample_rr(eng.ctx, count, 9, sid)
            assert tim.tim_get_profile(eng.ctx)["pass3_sets"] > 10
            off, mem, wid = tim.tim_get_rr(eng.ctx)
            roff, rmem, rwid = O.sample(og, 9, sid, count)
            assert np.array_equal(off, roff) and np.array_equal(wid, rwid)
            assert _sorted_sets(off, mem) == _sorted_sets(roff, rmem)
            assert tim.tim_kappa_sum(eng.ctx, 10, 9, sid, 5000) == O.kappa_sum(og, 10, 9, sid, 5000)
            seeds = np.array([0, 1, 2, 500], dtype=np.int32)
            assert tim.tim_covered_count(eng.ctx, seeds, 9, sid, count) == \
                O.covered_count(og, 9, sid, count, seeds)
