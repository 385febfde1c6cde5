"""The second pass's visited sets as bitmaps: node counts around a word of the bitmap, around the
sizes where it stops fitting the shared memory (per team size) and the hash's place in global
memory, sets from a few hundred members to beyond the pass's queue (8192), handed over from pass 1
and on to the heavy pass; independent cascade with every team size, triggering, and a batch.
Sets and widths equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
SID = O.make_sid(3, 0, 0)


def _compare(ctx, og, count):
    tim.tim_get_profile(ctx, reset=True)
    tim.tim_sample_rr(ctx, count, 4, SID)
    off, mem, wid = tim.tim_get_rr(ctx)
    roff, rmem, rwid = O.sample(og, 4, SID, count)
    assert np.array_equal(off, roff) and np.array_equal(wid, rwid)
    for j in range(count):
        assert np.array_equal(np.sort(mem[off[j]:off[j + 1]]), np.sort(rmem[roff[j]:roff[j + 1]]))
    return tim.tim_get_profile(ctx)["pass2_sets"]


# n / 32 + 1 words: 16 KB of shared memory per block for 8, 4, 2 and 1 teams, 200 KB for one,
# and 16384 words
NODES = [3000, 4095, 4096, 16351, 16352, 32735, 32736, 131039, 131040, 524287, 524288, 1638367,
         1638368]


@pytest.mark.parametrize("n", NODES)
def test_ic_teams(n):
    g = inputs.chain(n)
    w = inputs.constant(g, 0.9995)
    og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        for team in (0, 1, 2, 4, 8):
            tim.tim_set_team_size(eng.ctx, team)
            assert _compare(eng.ctx, og, 257) > 60


@pytest.mark.parametrize("n", [4096, 16351, 16352, 524287, 524288])
def test_triggering(n):
    g = inputs.chain(n)
    opts = inputs.triggering_all_in(g, 0.9995)
    og = O.load_graph_triggering(g.n, g.rowptr, g.dst, *opts)
    with tim.Engine(0) as eng:
        tim.tim_load_graph_triggering(eng.ctx, g.n, g.rowptr, g.dst, *opts)
        assert _compare(eng.ctx, og, 257) > 60


@pytest.mark.parametrize("scale", [10, 13])
def test_batch_of_unequal_graphs(scale):
    qs, engines, graphs = [], [], []
    for i, sc in enumerate((scale, 12)):
        g = inputs.rmat(sc, seed=60 + i)
        w = inputs.constant(g, 0.3)
        e = tim.Engine(0)
        tim.tim_load_graph(e.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        engines.append(e)
        graphs.append((g, w))
        qs.append(dict(ctx=e.ctx, k=4, eps=0.8, ell=1.0, tag=i + 1))
    out, _ = tim.tim_run_batch(qs, 9)
    for i, ((seeds, frac, st), (g, w)) in enumerate(zip(out, graphs)):
        og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
        ref = O.tim_plus(og, 4, 0.8, 1.0, 9, tag=i + 1)
        assert np.array_equal(seeds, ref.seeds) and st["covered"] == ref.covered
        assert st["theta"] == ref.theta
    for e in engines:
        e.close()
