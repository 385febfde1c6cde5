"""IC's first pass with several sets in flight per warp: set counts around the sets and the warps of
a launch, capacities of 128, 256 and 512 (an eighth of it per set), sets around these sizes that
move on with their state, an in-edge budget that stops them earlier, and lists under the skip rule
that are taken two at a time (and one at a time from 32768 in-edges). Sets, widths, kappa sums and
covered counts equal the oracle's, alone and in a batch."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
SID = O.make_sid(3, 0, 0)


def _compare(ctx, og, counts, seed=4):
    for count in counts:
        tim.tim_sample_rr(ctx, count, seed, SID)
        off, mem, wid = tim.tim_get_rr(ctx)
        roff, rmem, rwid = O.sample(og, seed, SID, count)
        assert np.array_equal(off, roff) and np.array_equal(wid, rwid)
        for j in range(count):
            assert np.array_equal(np.sort(mem[off[j]:off[j + 1]]),
                                  np.sort(rmem[roff[j]:roff[j + 1]]))
    return np.diff(roff)


@pytest.mark.parametrize("capacity", [128, 256, 512])
@pytest.mark.parametrize("name", ["rmat", "chain", "nothing", "everything"])
def test_counts_and_capacities(capacity, name):
    g = inputs.chain(5000) if name == "chain" else inputs.rmat(11, seed=71)
    w = inputs.constant(g, {"rmat": 0.05, "chain": 0.97, "nothing": 0.0, "everything": 1.0}[name])
    og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        tim.tim_set_pass1_capacity(eng.ctx, capacity)
        sizes = _compare(eng.ctx, og, (1, 7, 8, 9, 33, 2000))
        if name == "chain":  # on both sides of every capacity's share
            assert all(np.any(sizes == s) for s in (15, 16, 17, 32, 33, 64))
        many = 60_001  # more sets than the launch's warps hold at once
        assert tim.tim_kappa_sum(eng.ctx, 5, 4, SID, many) == O.kappa_sum(og, 5, 4, SID, many)
        seeds = np.array([0, 17, 300], dtype=np.int32)
        assert tim.tim_covered_count(eng.ctx, seeds, 4, SID, many) == \
            O.covered_count(og, 4, SID, many, seeds)
        tim.tim_set_width_budget(eng.ctx, 64)
        _compare(eng.ctx, og, (500,), seed=6)


def _hubs(d, hubs=16):
    """`hubs` nodes with d in-edges each from the leaves (probability 1.5 / d), every leaf with
    in-edges from three hubs (probability 1)."""
    r = np.random.Generator(np.random.Philox(5))
    leaves = np.arange(hubs, hubs + d)
    src = np.concatenate([np.tile(leaves, hubs)] + [(leaves * 7 + 5 * i) % hubs for i in range(3)])
    dst = np.concatenate([np.repeat(np.arange(hubs), d)] + [leaves] * 3)
    g = inputs.csr_from_pairs(hubs + d, src, dst)
    w = np.where(np.asarray(g.dst) < hubs, np.float32(1.5 / d), np.float32(1.0)).astype(np.float32)
    return g, w


@pytest.mark.parametrize("d", [511, 512, 513, 32767, 32768, 33000])
def test_lists_under_the_skip_rule(d):
    g, w = _hubs(d)
    og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        for team in (0, 1, 4):
            tim.tim_set_team_size(eng.ctx, team)
            sizes = _compare(eng.ctx, og, (3, 400))
            assert sizes.max() > 32
        seeds = np.array([1, 20], dtype=np.int32)
        assert tim.tim_covered_count(eng.ctx, seeds, 4, SID, 1500) == \
            O.covered_count(og, 4, SID, 1500, seeds)


def test_batch_of_many_small_queries():
    engines, graphs, qs = [], [], []
    for i in range(9):
        g = inputs.rmat(8 + i % 3, seed=80 + i)
        w = inputs.weighted_cascade(g)
        e = tim.Engine(0)
        tim.tim_load_graph(e.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        engines.append(e)
        graphs.append((g, w))
        qs.append(dict(ctx=e.ctx, k=3 + i, eps=0.6, ell=1.0, tag=i + 1))
    out, _ = tim.tim_run_batch(qs, 9)
    for i, ((seeds, frac, st), (g, w)) in enumerate(zip(out, graphs)):
        og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
        ref = O.tim_plus(og, 3 + i, 0.6, 1.0, 9, tag=i + 1)
        assert np.array_equal(seeds, ref.seeds) and st["covered"] == ref.covered
        assert st["kpt_star"] == ref.kpt.kpt_star and st["theta"] == ref.theta
    for e in engines:
        e.close()


@pytest.mark.parametrize("count", [2048, 2049])
def test_long_lists_of_few_and_many_sets(count):
    """Sets with coins in long in-lists of their own thresholds, on both sides of the number of
    sets from which on the heavy-set pass takes them earlier; more than 400,000 edges."""
    g = inputs.chung_lu(20_001, 500_000, 2.1, seed=8)
    assert g.m > 400_000
    w = inputs.trivalency(g, seed=2)
    sid = O.make_sid(1, 4, 0)
    off, _, wid = O.sample(O.load_graph(g.n, g.rowptr, g.dst, w, O.IC), 3, sid, count)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        tim.tim_sample_rr(eng.ctx, count, 3, sid)
        o, _, x = tim.tim_get_rr(eng.ctx)
        assert np.array_equal(o, off) and np.array_equal(x, wid)
