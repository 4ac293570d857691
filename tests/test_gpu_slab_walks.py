"""GPU parity of the kernels that walk a step's column list slab by slab (the
update of a local step before a round's last, and the gather that follows
it): one CTA or one warp per slab, with regions shorter and longer than one
pass of the group, against the oracle (1e-5 normwise per worker)."""
import numpy as np
import pytest

from oracle import rounds
from paper_1612_08608_gb300 import inputs
from parity import sparse_round_matching

pytestmark = pytest.mark.gpu


# d = 3,000 and 1,300,000 at N = 8: 94 slabs of 32 columns (one CTA each) and
# 1,270 of 1,024 (more than one wave of CTAs, so a warp per slab unless a region
# is long); the wide slabs' first region holds about 8 x cols distinct (worker,
# column) pairs: a few (one partial pass of a warp), about 1,000, and 2,100.
# Column 0 is in every row that is not empty, so that the shards are laid out as
# column lists at every size.
@pytest.mark.parametrize("d", [3000, 1300000])
@pytest.mark.parametrize("cols", [3, 128, 300])
def test_slab_walks_match_oracle(d, cols):
    from paper_1612_08608_gb300 import Context
    N, B, T, tau = 8, 64, 2, 2
    rng = np.random.default_rng(cols)
    sh = inputs.sparse_custom(seed=cols, N=N, d=cols, rows=4 * B, max_len=min(cols, 20), hot_col=0)
    for i in range(N):      # one column near the end, so that the last slab has a region of its own
        last = sh.rowptr[i][1:][np.diff(sh.rowptr[i]) > 0] - 1
        sh.col[i][last[rng.random(last.shape[0]) < 0.3]] = d - 1
    sh.d = d
    sched = rounds.graph_schedule("ring", N, 1)
    with Context(N, d, graph_seed=0, k=1) as ctx:
        ctx.set_model("logistic", batch=B, lr=0.3, l2=0.01)
        ctx.set_graph("ring")
        ctx.set_schedule(local_steps=tau)
        ctx.load_shards(sh)
        assert not ctx.debug_shard_layout()["entries"]
        W_t, _ = ctx.read_params()
        for t in range(T):
            ctx.round(1)
            W_n, _ = ctx.read_params()
            nbr, wgt = sched(t)
            err, lref, _ = sparse_round_matching(W_t.astype(np.float64), W_n, sh, t, B, "logistic", 0.3, nbr, wgt,
                                                 1e-5, l2=0.01, tau=tau)
            assert err <= 1e-5, (t, err)
            assert abs(ctx.read_metrics(t, 1)[0][0] - lref) <= 1e-5
            W_t = W_n
