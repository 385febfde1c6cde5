"""Workspaces that grow between calls start out clean even when the allocator returns the address
of the one they replace: few heavy sets first, many later, on one engine, with neighbouring buffers
of several sizes. RR set sizes and widths equal the oracle's."""
import ctypes

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


@pytest.mark.parametrize("counts", [(1, 4), (1, 2, 4), (2, 1, 3, 4)])
def test_growing_cascades(counts):
    """Cascades whose visited bitmaps (200,004 bytes each) sit in global memory, when the only
    hole that the allocator has for them holds other data: one bitmap and four start at the same
    address. Without live edges every cascade activates its seeds and nothing else."""
    n, k = 1_600_001, 1000
    seeds = np.random.default_rng(7).choice(n, k, replace=False).astype(np.int32)
    rowptr = np.ones(n + 1, dtype=np.int64)
    rowptr[0] = 0
    import torch
    torch.zeros(1, device="cuda")
    rt = ctypes.CDLL("libcudart.so.13")
    held = []

    def malloc(size):
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        held.append(p.value)
        return p.value

    try:
        with tim.Engine(0) as eng:
            tim.tim_load_graph(eng.ctx, n, rowptr, np.array([1], np.int32),
                               np.zeros(1, np.float32), tim.TIM_IC)
            # no hole of 200 KB left in the 2 MiB blocks that small allocations share, then one
            # of 1000 KB
            for _ in range(1000):
                if malloc(200 << 10) % (2 << 20) == 0:
                    break
            for _ in range(9):
                malloc(200 << 10)
            malloc(1000 << 10)
            hole = malloc(1000 << 10)
            assert rt.cudaMemset(ctypes.c_void_p(hole), 0xFF, ctypes.c_size_t(1000 << 10)) == 0
            torch.cuda.synchronize()
            held.remove(hole)
            assert rt.cudaFree(ctypes.c_void_p(hole)) == 0
            for count in counts:
                _, total, each = tim.tim_spread_mc(eng.ctx, seeds, count, 3, 0, want_counts=True)
                assert np.array_equal(each, np.full(count, k)) and total == count * k
    finally:
        for p in held:
            rt.cudaFree(ctypes.c_void_p(p))
