"""GPU parity of forward cascades where the kernel draws a cascade's whole world at once (live
bits over the out-records) beside walking its out-edges: worlds with more live edges than a
warp's stage holds, options of many in-edges, node counts around the shared-memory limits of
the visited bitmap, edge counts around the bit words, seeds whose cascades stay small.
Per-cascade counts equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
MC = O.make_sid(7, 0, 0)


def _check(eng, og, n, seeds, count, sid0=MC):
    mean, total, counts = tim.tim_spread_mc(eng.ctx, seeds, count, 23, sid0, want_counts=True)
    rc, rtot = O.spread_mc(og, seeds, count, 23, sid0)
    assert np.array_equal(counts.astype(np.int64), rc)
    assert total == rtot


@pytest.mark.parametrize("p", [1.0, 0.6, 0.02])
@pytest.mark.parametrize("m", [60_000, 60_003])
def test_dense_worlds(p, m):
    g = inputs.random_small(1500, m, seed=4)
    w = inputs.constant(g, p)
    og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        for seeds in ([7], list(range(0, 1500, 31))):
            _check(eng, og, g.n, seeds, 40)


@pytest.mark.parametrize("n", [127, 655_328, 655_360, 1_556_448, 1_556_480])
@pytest.mark.parametrize("model", ["ic", "lt"])
def test_bitmap_limits(n, model):
    g = inputs.chung_lu(n, 4 * n if n > 1000 else 500, seed=9)
    w = inputs.weighted_cascade(g) if model == "ic" else inputs.lt_random_normalised(g, 5)
    om = O.IC if model == "ic" else O.LT
    og = O.load_graph(g.n, g.rowptr, g.dst, w, om)
    deg = np.diff(g.rowptr)
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, om)
        _check(eng, og, n, np.argsort(-deg, kind="stable")[:20].tolist(), 8)
        _check(eng, og, n, [int(n - 1)], 8, MC + 100)  # walks only, or adds nothing


@pytest.mark.parametrize("kind", ["all_in", "random"])
def test_triggering_worlds(kind):
    g = inputs.rmat(11, seed=12)
    opts = (inputs.triggering_all_in(g, 0.5) if kind == "all_in"
            else inputs.triggering_random(g, 4, 40, seed=3))
    og = O.load_graph_triggering(g.n, g.rowptr, g.dst, *opts)
    with tim.Engine(0) as eng:
        tim.tim_load_graph_triggering(eng.ctx, g.n, g.rowptr, g.dst, *opts)
        for seeds in ([0, 1, 2, 3], [1777]):
            _check(eng, og, g.n, seeds, 300)
