"""The geometric-skip rule's digit thresholds T_b (tables computed at graph load): RR sets that
run through lists just under the rule's probability bound, with tiny probabilities, and of
lengths around powers of two equal the oracle's, which decides each digit by the 64 x 64-bit
product."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [512, 513, 1023, 1024, 1025, 4095, 4096, 20000])
def test_digit_thresholds(d):
    # hubs 0..3 with d in-edges each: p as large as the rule takes, 1/d, 2^-31 and 3 / d
    bl = d.bit_length()
    top = (2 ** 32 // (2 * bl + 2) - 1) / 2 ** 32
    ps = [top, 1.0 / d, 2.0 ** -31, min(3.0 / d, top)]
    src, dst, w = [], [], []
    for h, p in enumerate(ps):
        src += [4 + i for i in range(d)] + [(h + 1) % 4]
        dst += [h] * (d + 1)
        w += [p] * (d + 1)
    # every leaf is reached back from a hub, so that most RR sets run through several hubs
    for i in range(d):
        src.append(i % 4)
        dst.append(4 + i)
        w.append(1.0)
    order = np.lexsort((dst, src))
    src, dst = np.array(src)[order], np.array(dst, dtype=np.int32)[order]
    w = np.array(w, dtype=np.float32)[order]
    n = 4 + d
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=rowptr[1:])
    og = O.load_graph(n, rowptr, dst, w, O.IC)
    sid, count = O.make_sid(3, 0, 0), 4000
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, n, rowptr, dst, w, tim.TIM_IC)
        tim.tim_sample_rr(eng.ctx, count, 77, sid)
        off, mem, wid = tim.tim_get_rr(eng.ctx)
    roff, rmem, rwid = O.sample(og, 77, sid, count)
    assert np.array_equal(off, roff) and np.array_equal(wid, rwid)
    for j in range(count):
        assert np.array_equal(np.sort(mem[off[j]:off[j + 1]]), np.sort(rmem[roff[j]:roff[j + 1]]))
