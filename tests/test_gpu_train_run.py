"""Training in one cooperative launch: sample counts around the blocks of 32 samples and the
number of resident blocks, input widths from one to the largest. Split runs equal one run bit
for bit, each loss equals the loss tim_mlp_grad reports for the parameters at that step, and a
run larger than the resident blocks (one launch pair per step) starts with the same loss."""
import numpy as np
import pytest

from paper_1404_0900_gb300 import tim

pytestmark = pytest.mark.gpu


def _net(eng, d, seed):
    rng = np.random.default_rng(seed)
    net = tim.tim_mlp_create(eng.ctx, d)
    p = rng.uniform(-0.3, 0.3, tim.tim_mlp_param_count(net)).astype(np.float32)
    tim.tim_mlp_set_scaling(eng.ctx, net, rng.normal(size=d), 0.5 + rng.random(d), 1.5, 2.0)
    return net, p


@pytest.mark.parametrize("n,d", [(1, 12), (31, 12), (32, 1), (33, 12), (100, 5), (4863, 12),
                                 (4865, 12), (9728, 32), (9800, 12)])
def test_runs_split_and_match_the_gradient(n, d):
    rng = np.random.default_rng(n + d)
    x = rng.normal(size=(n, d)).astype(np.float32)
    y = rng.normal(size=n).astype(np.float32)
    with tim.Engine(0) as eng:
        net, p = _net(eng, d, 7)
        try:
            tim.tim_mlp_set_params(eng.ctx, net, p)
            whole = tim.tim_mlp_train(eng.ctx, net, x, y, 7, 1e-2)
            end = tim.tim_mlp_get_params(eng.ctx, net)
            tim.tim_mlp_set_params(eng.ctx, net, p)
            parts = []
            for steps in (3, 1, 3):
                loss, _ = tim.tim_mlp_grad(eng.ctx, net, x, y)
                h = tim.tim_mlp_train(eng.ctx, net, x, y, steps, 1e-2)
                assert h[0] == np.float32(loss)
                parts.append(h)
            assert np.array_equal(np.concatenate(parts), whole)
            assert np.array_equal(tim.tim_mlp_get_params(eng.ctx, net), end)
        finally:
            tim.tim_mlp_destroy(net)


@pytest.mark.parametrize("n,d", [(1, 1), (32, 12), (33, 5), (500, 32), (4865, 12), (9728, 12)])
def test_one_launch_equals_launches_per_step(n, d):
    # runs of one step are two launches, longer ones one
    rng = np.random.default_rng(3 * n + d)
    x = rng.normal(size=(n, d)).astype(np.float32)
    y = rng.normal(size=n).astype(np.float32)
    with tim.Engine(0) as eng:
        net, p = _net(eng, d, 9)
        try:
            out = []
            for runs in ((12,), (1,) * 12, (3, 1, 2, 6)):
                tim.tim_mlp_set_params(eng.ctx, net, p)
                before = tim.tim_launch_count(eng.ctx)
                h = np.concatenate([tim.tim_mlp_train(eng.ctx, net, x, y, s, 1e-2) for s in runs])
                out.append((h, tim.tim_mlp_get_params(eng.ctx, net)))
                launches = tim.tim_launch_count(eng.ctx) - before
                assert launches == sum(1 if s > 1 else 2 for s in runs)
            for h, q in out[1:]:
                assert np.array_equal(h, out[0][0]) and np.array_equal(q, out[0][1])
        finally:
            tim.tim_mlp_destroy(net)
