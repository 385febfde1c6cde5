"""Cascades of a known or oracle size around every line where their path changes: cascades that a
warp walks (at most 128 members and 1024 out-edges, calls of many cascades), rounds of at most 32
nodes, cascades of more than 4096 members, with the visited bitmap in the shared memory of half an
SM, of a whole one, and in global memory."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1404_0900_gb300 import inputs, tim

pytestmark = pytest.mark.gpu
MANY = 1300  # more than four times as many cascades as blocks at once


def _parts():
    """A forest: (name, layers) with layers[i] children in all per layer, each hanging off the
    layer before in turn; the root is layer 0."""
    parts = [(f"chain{n}", [1] * (n - 1)) for n in (1, 2, 127, 128, 129, 300)]
    parts += [(f"star{d}", [d]) for d in (31, 32, 33, 126, 127, 128, 1023, 1024, 1025)]
    parts += [(f"layers{a}", [a, a, 7, 5000, 3, 40]) for a in (4094, 4095, 4096, 4097)]
    parts += [("grows", [2, 5, 12, 30, 33, 70, 150, 400]), ("wave", [6000, 1, 6000, 2, 9000, 1])]
    return parts


@pytest.fixture(scope="module")
def forest():
    src, dst, roots, sizes = [], [], [], []
    n = 0
    for _, layers in _parts():
        level = np.array([n])
        roots.append(n)
        n += 1
        size = 1
        for width in layers:
            nodes = n + np.arange(width)
            src.append(level[np.arange(width) % len(level)])
            dst.append(nodes)
            n += width
            size += width
            level = nodes
        sizes.append(size)
    return n, np.concatenate(src), np.concatenate(dst), np.array(roots), np.array(sizes)


@pytest.mark.parametrize("model", [tim.TIM_IC, tim.TIM_LT])
@pytest.mark.parametrize("pad", [0, 700_001, 1_600_001])
def test_sizes_at_the_limits(forest, model, pad):
    """Every edge live: a cascade activates its tree, from the root and from roots together."""
    n, src, dst, roots, sizes = forest
    n = max(n, pad)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    order = np.argsort(src, kind="stable")
    np.cumsum(np.bincount(src, minlength=n), out=rowptr[1:])
    with tim.Engine(0) as eng:
        tim.tim_load_graph(eng.ctx, n, rowptr, dst[order].astype(np.int32),
                           np.ones(len(dst), np.float32), model)
        for seeds, size in [([r], s) for r, s in zip(roots, sizes)] + [
                (roots, sizes.sum()), (roots[:3], sizes[:3].sum()), ([roots[0]] * 70, sizes[0])]:
            for count in (3, MANY):
                _, total, counts = tim.tim_spread_mc(eng.ctx, np.array(seeds, np.int32), count, 5,
                                                     9, want_counts=True)
                assert total == count * size and np.all(counts == size)


@pytest.mark.parametrize("kind", ["wc", "p0.3", "lt", "trig"])
def test_many_small_cascades_equal_the_oracle(kind):
    g = inputs.chung_lu(2_001, 6_000, 2.1, seed=4)
    if kind == "trig":
        opts = inputs.triggering_random(g, seed=3)
        og = O.load_graph_triggering(g.n, g.rowptr, g.dst, *opts)
    else:
        w = (inputs.weighted_cascade(g) if kind == "wc" else inputs.constant(g, 0.3)
             if kind == "p0.3" else inputs.lt_random_normalised(g, seed=2))
        og = O.load_graph(g.n, g.rowptr, g.dst, w, O.LT if kind == "lt" else O.IC)
    seeds = np.random.default_rng(5).permutation(g.n).astype(np.int32)
    with tim.Engine(0) as eng:
        if kind == "trig":
            tim.tim_load_graph_triggering(eng.ctx, g.n, g.rowptr, g.dst, *opts)
        else:
            tim.tim_load_graph(eng.ctx, g.n, g.rowptr, g.dst, w,
                               tim.TIM_LT if kind == "lt" else tim.TIM_IC)
        for k in (1, 5, 33, 64, 65):
            want, total = O.spread_mc(og, seeds[:k], MANY, 7, 11)
            _, got, counts = tim.tim_spread_mc(eng.ctx, seeds[:k], MANY, 7, 11, want_counts=True)
            assert got == total and np.array_equal(counts, want)
