"""GPU parity of the list layout's local step with four, eight and twelve
consumer warps per CTA (GPU): shares just below and above what one tile of each
holds (1,024, 2,048 and 3,072 entries), and several tiles, against the oracle
round by round (1e-5 normwise per worker)."""
import numpy as np
import pytest

from oracle import rounds
from paper_1612_08608_gb300 import inputs
from parity import sparse_round_matching

pytestmark = pytest.mark.gpu


# 96 rows a minibatch over a worker's eight CTAs: 12 entries a CTA per entry of a row
@pytest.mark.parametrize("row_len", [1, 60, 64, 65, 100, 150, 171, 240, 257, 300, 500])
@pytest.mark.parametrize("loss", ["hinge", "logistic"])
def test_step_warps_match_oracle(row_len, loss):
    _check(4, 96, row_len, loss)


# many rows: shared memory leaves an SM two CTAs of eight warps, one of twelve, or one of eight; sixteen workers'
# clusters do not all fit at one CTA per SM
@pytest.mark.parametrize("N,B", [(16, 1024), (8, 2000), (16, 2048), (16, 2049)])
def test_step_warps_with_many_rows(N, B):
    _check(N, B, 40, "logistic")


def _check(N, B, row_len, loss):
    from paper_1612_08608_gb300 import Context
    d = 2000
    sh = inputs.sparse_custom(seed=row_len, N=N, d=d, rows=2 * B, hot_col=11,      # runs of 96: the list layout
                              lengths=[np.full(2 * B, row_len)] * N)
    sched = rounds.graph_schedule("ring", N, 1)
    W_t = (0.1 * np.random.default_rng(1).standard_normal((N, d))).astype(np.float32)
    with Context(N, d, graph_seed=0, k=1) as ctx:
        ctx.set_model(loss, batch=B, lr=0.2)
        ctx.set_graph("ring")
        ctx.load_shards(sh)
        ctx.write_params(W_t, 0)
        for t in range(3):
            ctx.round(1)
            W_n, _ = ctx.read_params()
            nbr, wgt = sched(t)
            err, lref, _ = sparse_round_matching(W_t.astype(np.float64), W_n, sh, t, B, loss, 0.2, nbr, wgt, 1e-5)
            assert err <= 1e-5, (t, err)
            lg = ctx.read_metrics(t, 1)[0][0]
            assert abs(lg - lref) <= 1e-5 * max(1.0, abs(lref)), (t, lg, lref)
            W_t = W_n
