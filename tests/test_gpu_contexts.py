"""Several contexts alive at once (GPU): one context's sizes do not disturb
another's launches, although both use the same kernels."""
import numpy as np
import pytest

from oracle import rounds
from paper_1612_08608_gb300 import inputs
from parity import sparse_round_matching

pytestmark = pytest.mark.gpu


def test_contexts_of_different_sizes_side_by_side():
    # minibatches of 600 and of 8 rows, long and short column lists: the
    # kernels' shared memory differs, the smaller context is set up last
    from paper_1612_08608_gb300 import Context
    made = []
    for N, d, B, max_len in [(8, 3000, 600, 60), (8, 3000, 8, 6)]:
        sh = inputs.sparse_custom(seed=B, N=N, d=d, rows=3 * B, max_len=max_len, hot_col=2)
        ctx = Context(N, d, graph_seed=0, k=1)
        ctx.set_model("logistic", batch=B, lr=0.3)
        ctx.set_graph("ring")
        ctx.load_shards(sh)
        ctx.round(1)
        made.append((ctx, sh, B))
    sched = rounds.graph_schedule("ring", 8, 1)
    for ctx, sh, B in made:
        W_t, _ = ctx.read_params()
        ctx.round(1)
        W_n, rnd = ctx.read_params()
        assert rnd == 2
        nbr, wgt = sched(1)
        err, _, _ = sparse_round_matching(W_t.astype(np.float64), W_n, sh, 1, B, "logistic", 0.3, nbr, wgt, 1e-5)
        assert err <= 1e-5
        ctx.close()


@pytest.mark.parametrize("residency", ["device", "host"])
def test_setup_behind_queued_work_of_the_default_stream(residency):
    # the context's streams do not wait for the legacy default stream: nothing that a context sets up may be queued
    # there, behind the caller's own work, and land after the first round's copies and kernels
    import torch
    from paper_1612_08608_gb300 import Context
    N, d, B = 6, 8000, 32
    rng = np.random.default_rng(1)
    W0 = rng.standard_normal((N, d)).astype(np.float32)
    sh = inputs.sparse_custom(seed=3, N=N, d=d, rows=4 * B, max_len=40)
    dev = torch.from_numpy(W0).cuda()
    torch.cuda.synchronize()
    made = []
    torch.cuda._sleep(400_000_000)                     # about 0.2 s of the default stream
    for model in (False, True):
        ctx = Context(N, d, graph_seed=0, k=N - 1)     # complete graph: no table is uploaded
        ctx.set_graph("complete")
        if model:
            ctx.set_model("logistic", batch=B, lr=0.3)
            ctx.set_shard_residency(residency)
            ctx.load_shards(sh)
            ctx.write_params(W0, 0)
        else:
            ctx.write_params_device(dev, 0)
        ctx.round(1)
        made.append(ctx)
    torch.cuda.synchronize()                           # whatever was queued late has run
    mean = W0.astype(np.float64).mean(axis=0)
    got, rnd = made[0].read_params()
    assert rnd == 1 and np.abs(got - mean).max() <= 1e-6 * np.abs(mean).max()
    sched = rounds.graph_schedule("complete", N, N - 1)
    W_t = W0
    for t in range(3):
        if t:
            made[1].round(1)
        W_n, _ = made[1].read_params()
        nbr, wgt = sched(t)
        err, lref, _ = sparse_round_matching(W_t.astype(np.float64), W_n, sh, t, B, "logistic", 0.3, nbr, wgt, 1e-5)
        assert err <= 1e-5, (t, err)
        assert abs(made[1].read_metrics(t, 1)[0][0] - lref) <= 1e-5
        W_t = W_n
    for ctx in made:
        ctx.close()


@pytest.mark.parametrize("N,d", [(3, 100), (16, 200001)])
def test_device_parameters_still_being_made_on_the_default_stream(N, d):
    # parameters that the default stream is yet to fill when they are handed over
    import torch
    from paper_1612_08608_gb300 import Context
    want = np.random.default_rng(N).standard_normal((N, d)).astype(np.float32)
    src = torch.from_numpy(want).cuda()
    with Context(N, d, graph_seed=0, k=1) as ctx:
        dev = torch.zeros_like(src)
        torch.cuda.synchronize()
        torch.cuda._sleep(200_000_000)                 # about 0.1 s
        dev.copy_(src)
        ctx.write_params_device(dev, 4)
        got, rnd = ctx.read_params()
    assert rnd == 4 and np.array_equal(got, want)
