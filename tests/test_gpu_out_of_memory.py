"""Calls that run out of device memory at any of their allocations (a limit on what the context
holds stands in for a full device): TIM_ERR_OOM, an empty RR-set store, and a context whose next
calls are right. RR sets equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
FREE = 2 ** 64 - 1


def _case(model):
    g = inputs.chung_lu(3_001, 30_000, 2.1, seed=3)
    if model == tim.TIM_IC:
        w = inputs.weighted_cascade(g)
    else:
        w = inputs.lt_random_normalised(g, seed=4)
    return g, w, O.load_graph(g.n, g.rowptr, g.dst, w, model)


def _load(eng, g, w, model):
    tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, model)


def _sorted(off, mem):
    return [np.sort(mem[off[i]:off[i + 1]]) for i in range(len(off) - 1)]


@pytest.mark.parametrize("model", [tim.TIM_IC, tim.TIM_LT])
def test_sampling_without_room(model):
    g, w, og = _case(model)
    sid, few, many = O.make_sid(1, 5, 0), 500, 100_000
    off, mem, wid = O.sample(og, 3, sid, many)
    sets = _sorted(off, mem)

    def check(eng, count):
        o, m, x = tim.tim_get_rr(eng.ctx)
        assert np.array_equal(o, off[:count + 1]) and np.array_equal(x, wid[:count])
        assert all(np.array_equal(a, b) for a, b in zip(_sorted(o, m), sets))

    with tim.Engine(0) as eng:
        _load(eng, g, w, model)
        tim.tim_sample_rr(eng.ctx, many, 3, sid)
        full = tim.tim_memory_held(eng.ctx)
    failed = 0
    with tim.Engine(0) as eng:
        _load(eng, g, w, model)
        tim.tim_sample_rr(eng.ctx, few, 3, sid)
        first = tim.tim_memory_held(eng.ctx)
        assert first < full
        for limit in np.linspace(first, full, 60).astype(np.int64):
            tim.tim_sample_rr(eng.ctx, few, 3, sid)
            tim.tim_kpt_estimate(eng.ctx, 3, 1.0, 3)
            tim.tim_sample_rr(eng.ctx, few, 3, sid)
            tim.tim_set_memory_limit(eng.ctx, int(limit))
            try:
                tim.tim_sample_rr(eng.ctx, many, 3, sid)
                check(eng, many)
            except tim.TimError as e:
                assert e.code == tim.TIM_ERR_OOM
                failed += 1
                assert tim.tim_rr_size(eng.ctx) == (0, 0)
            tim.tim_set_memory_limit(eng.ctx, FREE)
            if tim.tim_rr_size(eng.ctx) == (0, 0):
                assert not tim.tim_coverage_counts(eng.ctx, g.n).any()
                seeds, _, cov = tim.tim_node_select(eng.ctx, 3)
                assert seeds.tolist() == [0, 1, 2] and cov == 0
                with pytest.raises(tim.TimError):
                    tim.tim_refine_kpt(eng.ctx, 3, 1.0, 0.3, 3)
                tim.tim_sample_rr(eng.ctx, few, 3, sid)
                check(eng, few)
        tim.tim_sample_rr(eng.ctx, many, 3, sid)
        check(eng, many)
    assert failed > 0


def test_steps_after_a_selection_without_room():
    g, w, og = _case(tim.TIM_IC)
    sid = O.make_sid(1, 5, 0)
    off, mem, _ = O.sample(og, 3, sid, 2000)
    counts = np.bincount(mem, minlength=g.n)
    v = int(np.argmax(counts))
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        tim.tim_sample_rr(eng.ctx, 2000, 3, sid)
        tim.tim_select_begin(eng.ctx)
        tim.tim_set_memory_limit(eng.ctx, 0)
        with pytest.raises(tim.TimError):
            tim.tim_node_select(eng.ctx, g.n)
        tim.tim_set_memory_limit(eng.ctx, FREE)
        assert np.array_equal(tim.tim_select_counts(eng.ctx, g.n), counts)
        assert tim.tim_select_take(eng.ctx, v) == counts[v]


@pytest.mark.parametrize("ell,dense", [(1.0, False), (20.0, False), (1.0, True), (8000.0, True)])
def test_algorithm_2_in_the_memory_of_its_largest_round(ell, dense):
    """Several rounds in one call are for speed only: in the memory that its rounds take one
    after another Algorithm 2 gives the same estimate and leaves the same store."""
    k, seed = 2, 3
    if dense:  # stops in round 1 or 2
        g = inputs.complete(60)
        w = inputs.constant(g, 0.5)
    else:
        g = inputs.chung_lu(3_001, 12_000, 2.1, seed=3)
        w = inputs.constant(g, 0.01)
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        want = tim.tim_kpt_estimate(eng.ctx, k, ell, seed)
        off, mem, wid = tim.tim_get_rr(eng.ctx)
    last = want[1] or O.kpt_rounds(g.n)
    assert (last <= 2) == dense
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        for i in range(1, last + 1):
            tim.tim_sample_rr(eng.ctx, O.c_i(g.n, ell, i), seed, O.make_sid(1, i, 0))
        room = tim.tim_memory_held(eng.ctx)
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        tim.tim_set_memory_limit(eng.ctx, room + (64 << 10))
        assert tim.tim_kpt_estimate(eng.ctx, k, ell, seed) == want
        o, m, x = tim.tim_get_rr(eng.ctx)
        assert np.array_equal(o, off) and np.array_equal(x, wid)
        assert all(np.array_equal(a, b) for a, b in zip(_sorted(o, m), _sorted(off, mem)))


def test_the_second_store_makes_room():
    """What Algorithm 2 keeps for its grouped rounds does not take memory from a larger call."""
    g, w, og = _case(tim.TIM_IC)
    sid, count = O.make_sid(1, 5, 0), 60_000
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        tim.tim_sample_rr(eng.ctx, count, 3, sid)
        off, mem, _ = tim.tim_get_rr(eng.ctx)
        room = tim.tim_memory_held(eng.ctx)
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        tim.tim_kpt_estimate(eng.ctx, 2, 1.0, 3)
        tim.tim_set_memory_limit(eng.ctx, room + (64 << 10))
        tim.tim_sample_rr(eng.ctx, count, 3, sid)
        o, m, _ = tim.tim_get_rr(eng.ctx)
        assert np.array_equal(o, off)
        assert all(np.array_equal(a, b) for a, b in zip(_sorted(o, m), _sorted(off, mem)))


@pytest.mark.parametrize("k", [1, 40])
def test_selection_in_the_memory_of_the_full_index(k):
    """The greedy over candidates gives way to the full index where it has no room."""
    g, w, og = _case(tim.TIM_IC)
    sid, count = O.make_sid(1, 5, 0), 60_000
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        tim.tim_sample_rr(eng.ctx, count, 3, sid)
        tim.tim_select_begin(eng.ctx)  # an open selection keeps to the full index
        want = tim.tim_node_select(eng.ctx, k)
        room = tim.tim_memory_held(eng.ctx)
    with tim.Engine(0) as eng:
        _load(eng, g, w, tim.TIM_IC)
        tim.tim_sample_rr(eng.ctx, count, 3, sid)
        tim.tim_set_memory_limit(eng.ctx, room + (4 << 10))
        got = tim.tim_node_select(eng.ctx, k)
        assert np.array_equal(got[0], want[0]) and got[1:] == want[1:]
        tim.tim_set_memory_limit(eng.ctx, FREE)
        got = tim.tim_node_select(eng.ctx, k)
        assert np.array_equal(got[0], want[0]) and got[1:] == want[1:]
    off, mem, _ = O.sample(og, 3, sid, count)
    assert np.array_equal(want[0], O.greedy(g.n, off, mem, k)[0])


@pytest.mark.parametrize("model", [tim.TIM_IC, tim.TIM_LT])
def test_cascades_without_room_for_worlds(model):
    """Cascades need the out-records, a queue per block and the counts; whole worlds (the
    out-record of every in-edge, a bit per out-record and block) only where there is room."""
    g, w, og = _case(model)
    count, seeds = 400, np.arange(30, dtype=np.int32)
    counts, total = O.spread_mc(og, seeds, count, 3, 0)
    with tim.Engine(0) as eng:
        _load(eng, g, w, model)
        one = tim.tim_spread_mc(eng.ctx, seeds, count, 3, 0, want_counts=True)
        full = tim.tim_memory_held(eng.ctx)
    with tim.Engine(0) as eng:
        _load(eng, g, w, model)
        blocks = min(count, 2 * 160)
        room = tim.tim_memory_held(eng.ctx) + 4 * blocks * g.n + 12 * (g.n + 1) + 8 * g.m + 4 * count
        assert room + (64 << 10) < full
        tim.tim_set_memory_limit(eng.ctx, room + (64 << 10))
        for _ in range(2):
            got = tim.tim_spread_mc(eng.ctx, seeds, count, 3, 0, want_counts=True)
            assert got[1] == one[1] == total
            assert np.array_equal(got[2], counts) and np.array_equal(one[2], counts)
        tim.tim_set_memory_limit(eng.ctx, FREE)
        _load(eng, g, w, model)
        got = tim.tim_spread_mc(eng.ctx, seeds, count, 3, 0, want_counts=True)
        assert got[1] == total and np.array_equal(got[2], counts)
