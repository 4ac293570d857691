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
