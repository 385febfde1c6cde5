"""Workspaces that grow between calls start out clean even when the allocator returns the address
of the one they replace: few heavy sets first, many later, on one engine, with neighbouring buffers
of several sizes. RR set sizes and widths equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    g = inputs.chung_lu(20_001, 500_000, 2.1, seed=23)
    w = inputs.trivalency(g, seed=4)
    og = O.load_graph(g.n, g.rowptr, g.dst, w, O.IC)
    sid = O.make_sid(1, 13, 0)
    off, _, wid = O.sample(og, 3, sid, 200_000)
    return g, w, np.diff(off), wid, sid


@pytest.mark.parametrize("capacity", [128, 256, 512])
@pytest.mark.parametrize("counts", [(200_000,), (700, 200_000), (100, 1500, 20_000, 200_000)])
def test_growing_calls(case, capacity, counts):
    g, w, sizes, widths, sid = case
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w, tim.TIM_IC)
        tim.tim_set_pass1_capacity(eng.ctx, capacity)
        tim.tim_kpt_estimate(eng.ctx, 1, 1.0, 3)
        for count in counts:
            tim.tim_sample_rr(eng.ctx, count, 3, sid)
            off, _, wid = tim.tim_get_rr(eng.ctx)
            assert np.array_equal(np.diff(off), sizes[:count])
            assert np.array_equal(wid, widths[:count])
