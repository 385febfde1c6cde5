"""LT chains in pass 1 with lanes handled in groups: set counts around the lanes of a warp and of
the group that is handled together, chains around the pass's capacity of 1024 members (longer
ones move on), chains that end in long cycles (revisits far back), single and batched queries.
Sets, widths, kappa sums and covered counts equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
SID = O.make_sid(3, 0, 0)


def _graph(name):
    if name == "rmat":
        return inputs.rmat(12, seed=51)
    if name.startswith("chain"):
        return inputs.chain(int(name[5:]))
    if name.startswith("cycle"):
        return inputs.cycle(int(name[5:]))
    raise KeyError(name)


@pytest.mark.parametrize("name", ["rmat", "chain1023", "chain1025", "chain1400", "cycle1023",
                                  "cycle1024", "cycle1025", "cycle300"])
def test_lanes(name):
    g = _graph(name)
    w = inputs.lt_random_normalised(g, 6) if name == "rmat" else inputs.lt_inverse_indegree(g)
    og = O.load_graph(g.n, g.rowptr, g.dst, w, O.LT)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_LT)
        for count in (1, 7, 8, 9, 31, 33, 3001):
            tim.tim_sample_rr(eng.ctx, count, 4, SID)
            off, mem, wid = tim.tim_get_rr(eng.ctx)
            roff, rmem, rwid = O.sample(og, 4, SID, count)
            assert np.array_equal(off, roff) and np.array_equal(wid, rwid)
            for j in range(count):
                assert np.array_equal(np.sort(mem[off[j]:off[j + 1]]),
                                      np.sort(rmem[roff[j]:roff[j + 1]]))
        assert tim.tim_kappa_sum(eng.ctx, 5, 4, SID, 3001) == O.kappa_sum(og, 5, 4, SID, 3001)
        seeds = np.array([0, 17], dtype=np.int32)
        assert tim.tim_covered_count(eng.ctx, seeds, 4, SID, 3001) == \
            O.covered_count(og, 4, SID, 3001, seeds)


def test_batched_lanes():
    g = inputs.rmat(11, seed=52)
    w = inputs.lt_random_normalised(g, 6)
    c = inputs.cycle(1100)
    wc = inputs.lt_inverse_indegree(c)
    with tim.Engine(0) as e1, tim.Engine(0) as e2:
        tim.tim_load_graph(e1.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_LT)
        tim.tim_load_graph(e2.ctx, c.n, c.rowptr, c.dst, wc, tim.TIM_LT)
        qs = [dict(ctx=e1.ctx, k=5, eps=0.5, ell=1.0, tag=1),
              dict(ctx=e2.ctx, k=3, eps=0.5, ell=1.0, tag=2)]
        out, _ = tim.tim_run_batch(qs, 9)
    for (seeds, frac, st), (gr, wt), k, tag in zip(out, ((g, w), (c, wc)), (5, 3), (1, 2)):
        og = O.load_graph(gr.n, gr.rowptr, gr.dst, wt, O.LT)
        ref = O.tim_plus(og, k, 0.5, 1.0, 9, tag=tag)
        assert np.array_equal(seeds, ref.seeds) and st["covered"] == ref.covered
        assert st["kpt_star"] == ref.kpt.kpt_star and st["theta"] == ref.theta
