"""tim_node_select_noalloc at the sizes where its single launch can go wrong: one node, no sets,
one set, sets longer than the lanes that share one, node counts around the blocks' ranges, hub
members, k up to its limit; members and offsets out of range are still refused."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _select(n, off, mem, k):
    import torch
    from paper_1404_0900_gb300 import tim
    d_off = torch.from_numpy(np.asarray(off, dtype=np.int64)).cuda()
    d_mem = torch.from_numpy(np.asarray(mem, dtype=np.int32)).cuda()
    d_seeds = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    d_cov = torch.zeros(1, dtype=torch.int64, device="cuda")
    tim.tim_node_select_noalloc(0, None, n, len(off) - 1, d_off, d_mem, k, d_seeds, d_cov)
    return d_seeds.cpu().numpy(), int(d_cov.item())


def _store(n, sizes, seed, skew=3.0):
    r = np.random.default_rng(seed)
    sets = [np.unique((n * r.random(s) ** skew).astype(np.int64)) for s in sizes]
    off = np.concatenate([[0], np.cumsum([len(s) for s in sets])])
    return off, np.concatenate(sets) if sets else np.zeros(0, dtype=np.int64)


@pytest.mark.parametrize("n,sizes,k", [
    (1, [1, 1, 1], 1), (5, [], 3), (2, [1], 2), (77, [1] * 500, 77),
    (1023, [300] * 40 + [1] * 2000, 60), (1024, [9] * 3000, 1024), (1025, [8] * 3000, 10),
    (155_649, [6] * 30_000, 50), (262_144, [40] * 3000, 25)])
def test_sizes(n, sizes, k):
    off, mem = _store(n, sizes, n)
    seeds, cov = _select(n, off, mem, k)
    rseeds, rcov, _ = O.greedy(n, off, mem, k)
    assert np.array_equal(seeds, rseeds) and cov == rcov


def test_out_of_range_is_refused_and_the_next_call_is_right():
    from paper_1404_0900_gb300 import tim
    off, mem = _store(500, [5] * 300, 3)
    for bad in (-1, 500):
        m = mem.copy()
        m[17] = bad
        with pytest.raises(tim.TimError) as ei:
            _select(500, off, m, 4)
        assert ei.value.code == -1
    o = off.copy()
    o[10] = o[12] + 1  # a set whose end lies before its start
    with pytest.raises(tim.TimError):
        _select(500, o, mem, 4)
    rseeds, rcov, _ = O.greedy(500, off, mem, 4)
    seeds, cov = _select(500, off, mem, 4)
    assert np.array_equal(seeds, rseeds) and cov == rcov
