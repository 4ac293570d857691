"""GPU parity of the entry layout (columns spread evenly over the reduce's
slabs: products exported by the reduce, row sums, updates from the rows' r
inside the reduce) against the oracle, round by round (1e-5 normwise per
worker), at the edges of its row passes, runs and regions, and on both sides
of the rule that chooses it."""
import numpy as np
import pytest

from oracle import rounds
from paper_1612_08608_gb300 import inputs
from parity import sparse_round_matching

pytestmark = pytest.mark.gpu


def _uses_entries(ctx):
    return ctx.debug_shard_layout()["entries"]


def _make(sh, N, k, kind, loss, B, lr, l2=0.0, tau=1, residency="device", sync="bsp", regen=False):
    from paper_1612_08608_gb300 import Context
    ctx = Context(N, sh.d, graph_seed=7, k=k)
    ctx.set_model(loss, batch=B, lr=lr, l2=l2)
    ctx.set_graph(kind, regenerate=regen)
    ctx.set_schedule(local_steps=tau)
    ctx.set_shard_residency(residency)
    ctx.set_sync_mode(sync)
    ctx.load_shards(sh)
    return ctx


def _check(ctx, sh, T, B, loss, lr, sched, l2=0.0, tau=1, W0=None):
    if W0 is not None:
        ctx.write_params(W0, 0)
    W_t, _ = ctx.read_params()
    for t in range(T):
        ctx.round(1)
        W_n, _ = ctx.read_params()
        nbr, wgt = sched(t)
        err, lref, cref = sparse_round_matching(W_t.astype(np.float64), W_n, sh, t, B, loss, lr, nbr, wgt, 1e-5,
                                                l2=l2, tau=tau)
        assert err <= 1e-5, (t, err)
        lg, cg = ctx.read_metrics(t, 1)
        assert abs(lg[0] - lref) <= 1e-5 * max(1.0, abs(lref)), (t, lg[0], lref)
        assert abs(cg[0] - cref) <= 1e-4 * cref + 1e-6 * np.abs(W_n).max() * np.sqrt(W_n.size)
        W_t = W_n


# rows of a CTA's pass are 32: minibatches of 1, 31, 33 and 100 rows; rows of 0 to 260 entries (eight lanes
# cover 32 places a load and 128 a pass)
@pytest.mark.parametrize("B", [1, 31, 33, 100])
@pytest.mark.parametrize("N,k,kind", [(1, 0, "identity"), (3, 1, "ring"), (9, 2, "root"), (7, 5, "random_regular"),
                                      (6, 5, "complete")])
def test_rows_and_graphs(B, N, k, kind):
    d = 160003
    rng = np.random.default_rng(B)
    edge = np.array([0, 1, 3, 4, 5, 31, 32, 33, 127, 128, 129, 260])
    # every length occurs; most rows are 100 to 260 long, so that padding to 260 wastes little
    lengths = [np.where(rng.random(3 * B) < 0.4, rng.choice(edge, 3 * B), rng.integers(100, 261, 3 * B))
               for _ in range(N)]
    for ln in lengths:
        ln[0] = 200
    sh = inputs.sparse_custom(seed=B, N=N, d=d, rows=3 * B, lengths=lengths)
    W0 = (0.1 * rng.standard_normal((N, d))).astype(np.float32)
    with _make(sh, N, k, kind, "logistic", B, 0.5, regen=kind == "random_regular") as ctx:
        assert _uses_entries(ctx)
        sched = rounds.graph_schedule(kind, N, k, graph_seed=7, regenerate=kind == "random_regular")
        _check(ctx, sh, 4, B, "logistic", 0.5, sched, W0=W0)


@pytest.mark.parametrize("residency", ["device", "host"])
@pytest.mark.parametrize("sync", ["bsp", "notify_ack"])
def test_local_steps_l2_and_residency(residency, sync):
    N, d, B, tau = 10, 30011, 48, 3
    sh = inputs.sparse_custom(seed=2, N=N, d=d, rows=7 * B, max_len=40)
    sched = rounds.graph_schedule("random_regular", N, 3, graph_seed=7, regenerate=True)
    with _make(sh, N, 3, "random_regular", "hinge", B, 0.4, l2=0.02, tau=tau, residency=residency, sync=sync,
               regen=True) as ctx:
        assert _uses_entries(ctx)
        _check(ctx, sh, 3, B, "hinge", 0.4, sched, l2=0.02, tau=tau)


# The longest run a column may have is 32 entries and the longest region 704: on either side of both the rounds
# match the oracle, and the layout changes where the rule says.
@pytest.mark.parametrize("hot_rows,entries", [(1, True), (2, True), (31, True), (32, True), (33, False), (64, False)])
def test_runs_up_to_the_rule(hot_rows, entries):
    N, d, B = 4, 4000, 64
    rng = np.random.default_rng(hot_rows)
    sh = inputs.sparse_custom(seed=hot_rows, N=N, d=d, rows=2 * B, lengths=[np.full(2 * B, 12)] * N)
    for i in range(N):
        sh.col[i] += 1 - (sh.col[i] == d - 1)              # column 0 unused, the last kept inside
        for t in range(2):
            for b in rng.choice(B, hot_rows, replace=False):
                sh.col[i][sh.rowptr[i][t * B + b]] = 0
        for r in range(2 * B):                             # distinct within a row still
            a, e = sh.rowptr[i][r], sh.rowptr[i][r + 1]
            u = np.unique(sh.col[i][a:e])
            while u.shape[0] < e - a:
                u = np.unique(np.concatenate([u, rng.integers(1, d, 1).astype(np.int32)]))
            sh.col[i][a:e] = u
    with _make(sh, N, 2, "root", "logistic", B, 0.5) as ctx:
        assert _uses_entries(ctx) == entries
        _check(ctx, sh, 4, B, "logistic", 0.5, rounds.graph_schedule("root", N, 2))


@pytest.mark.parametrize("per_row,entries", [(8, True), (10, True), (11, False)])
def test_regions_up_to_the_rule(per_row, entries):
    # 313 slabs of 1,024 columns (N = 8); the first holds 64 rows x per_row entries of worker 0, and about 15 entries of
    # padding at 640 (before runs that would cross a multiple of 32)
    N, d, B = 8, 320000, 64
    ln = [np.full(2 * B, per_row)] + [np.zeros(2 * B, np.int64)] * (N - 1)
    sh = inputs.sparse_custom(seed=per_row, N=N, d=1024, rows=2 * B, lengths=ln)
    sh.d = d
    with _make(sh, N, 1, "ring", "logistic", B, 0.5) as ctx:
        assert _uses_entries(ctx) == entries
        _check(ctx, sh, 3, B, "logistic", 0.5, rounds.graph_schedule("ring", N, 1))


def test_empty_minibatches_and_two_runs_bit_identical():
    N, d, B = 5, 5000, 40
    rng = np.random.default_rng(0)
    lengths = [rng.integers(0, 60, 3 * B) for _ in range(N)]
    for ln in lengths:
        ln[B:2 * B] = 0
    sh = inputs.sparse_custom(seed=9, N=N, d=d, rows=3 * B, lengths=lengths)
    outs = []
    for mode in ("bsp", "bsp", "notify_ack"):
        with _make(sh, N, 1, "ring", "logistic", B, 0.5, sync=mode) as ctx:
            assert _uses_entries(ctx)
            ctx.round(7)
            outs.append((ctx.read_params()[0], ctx.read_metrics(0, 7)))
    for W, (lm, cm) in outs[1:]:
        assert np.array_equal(W, outs[0][0]) and np.array_equal(lm, outs[0][1][0]) and np.array_equal(cm, outs[0][1][1])
    assert abs(outs[0][1][0][1] - np.log(2.0)) <= 1e-6    # minibatch 1 is empty: the loss of m = 0


# Updates between local steps either stream the slabs (one parameter in 24 or more touched) or touch parameters
# one by one: 21 workers x 30,011 columns with about 75,000 entries a minibatch, and with about 13,000; a ragged
# last slab, columns in the first and last place, runs of several rows.
@pytest.mark.parametrize("residency", ["device", "host"])
@pytest.mark.parametrize("kind,k", [("root", 2), ("complete", 20)])
@pytest.mark.parametrize("max_len,streams", [(300, True), (50, False)])
def test_local_steps_streamed_and_touched(kind, k, residency, max_len, streams):
    N, d, B, tau, lr, l2 = 21, 30011, 24, 3, 0.4, 0.02
    sh = inputs.sparse_custom(seed=8, N=N, d=d, rows=7 * B, max_len=max_len)
    for i in range(N):
        ends = sh.rowptr[i][1:][np.diff(sh.rowptr[i]) > 1] - 1
        sh.col[i][ends[::3]] = d - 1
        starts = sh.rowptr[i][:-1][np.diff(sh.rowptr[i]) > 1]
        sh.col[i][starts[::5]] = 0
    rng = np.random.default_rng(3)
    W0 = (0.1 * rng.standard_normal((N, d))).astype(np.float32)
    with _make(sh, N, k, kind, "logistic", B, lr, l2=l2, tau=tau, residency=residency) as ctx:
        assert ctx.debug_shard_layout()["streams"] == streams
        before = ctx.kernel_launches()
        _check(ctx, sh, 2, B, "logistic", lr, rounds.graph_schedule(kind, N, k, graph_seed=7), l2=l2, tau=tau, W0=W0)
        # one gather at the start; per round tau steps, tau - 1 updates (and gathers, unless streamed), a reduce
        assert ctx.kernel_launches() - before == 1 + 2 * (2 * tau if streams else 3 * tau - 1)


@pytest.mark.parametrize("B,row_len,packed", [(512, 128, True), (512, 129, False), (513, 128, False), (2, 4000, True),
                                              (1, 5000, True), (1024, 64, True), (1025, 64, False)])
def test_row_and_place_in_the_code(B, row_len, packed):
    # row and place share 16 bits where they fit: bits of the row + bits of the place <= 16
    N, d = 2, 600011
    sh = inputs.sparse_custom(seed=B, N=N, d=d, rows=2 * B, lengths=[np.full(2 * B, row_len)] * N)
    W0 = (0.1 * np.random.default_rng(2).standard_normal((N, d))).astype(np.float32)
    with _make(sh, N, 1, "complete", "logistic", B, 0.5, tau=2) as ctx:
        assert ctx.debug_shard_layout()["entry_bytes"] == (8 if packed else 10)
        _check(ctx, sh, 2, B, "logistic", 0.5, rounds.graph_schedule("complete", N, 1), tau=2, W0=W0)


@pytest.mark.parametrize("B,halves", [(2, False), (24, False), (24, True)])
def test_notify_ack_after_streamed_local_steps_equals_bsp(B, halves):
    # a gated reduce starts while the round's last local step runs, and reads parameters that the step before has
    # updated by streaming the slabs; `halves`: a round's steps touch one half of the columns each, so that the reduce
    # has no worker to wait for in the slabs that the streamed update has written
    N, d = 21, 30011 if B == 24 else 2003
    sh = inputs.sparse_custom(seed=4, N=N, d=d, rows=6 * B, max_len=300)
    if halves:
        half = d // 2
        for i in range(N):
            for r in range(6 * B):
                a, e = sh.rowptr[i][r:r + 2]
                c = np.random.default_rng(1000 * i + r).choice(half, e - a, replace=False)
                sh.col[i][a:e] = np.sort(c) + (half if (r // B) % 2 else 0)
    outs = []
    for sync in ("bsp", "notify_ack"):
        with _make(sh, N, 2, "root", "logistic", B, 0.4, l2=0.02, tau=2, sync=sync) as ctx:
            before = ctx.kernel_launches()
            ctx.round(40)
            outs.append((ctx.read_params()[0], ctx.read_metrics(0, 40)))
            assert ctx.kernel_launches() - before == 1 + 40 * 4      # streamed: two steps, one update, one reduce
    assert np.array_equal(outs[0][0], outs[1][0])
    assert np.array_equal(outs[0][1][0], outs[1][1][0]) and np.array_equal(outs[0][1][1], outs[1][1][1])


# A reduce that finds a flag missing passes its slabs on unwritten, and its entry ring with them: one slab a CTA,
# and eight (the ring's six slots are used again)
@pytest.mark.parametrize("sync", ["bsp", "notify_ack"])
@pytest.mark.parametrize("N,d,max_len", [(6, 2003, 30), (8, 1300000, 300)])
def test_missing_notify_and_the_rounds_after_it(N, d, max_len, sync):
    from paper_1612_08608_gb300 import AsapError
    B = 32
    sh = inputs.sparse_custom(seed=5, N=N, d=d, rows=4 * B, max_len=max_len)
    W0 = (0.1 * np.random.default_rng(2).standard_normal((N, d))).astype(np.float32)
    outs = []
    for stall in (False, True):
        with _make(sh, N, 1, "ring", "logistic", B, 0.4, sync=sync) as ctx:
            assert _uses_entries(ctx)
            ctx.write_params(W0, 0)
            if stall:
                for _ in range(3):
                    ctx.set_wait_limit_ns(5_000_000)
                    ctx.debug_skip_notify(N - 2)
                    ctx.round(1)
                    with pytest.raises(AsapError) as ei:
                        ctx.sync()
                    assert ei.value.name == "ASAP_ERR_TIMEOUT"
                    ctx.write_params(W0, 0)
                ctx.set_wait_limit_ns(200_000_000)
            ctx.round(3)
            outs.append((ctx.read_params()[0], ctx.read_metrics(0, 3)))
    assert np.array_equal(outs[0][0], outs[1][0])
    assert np.array_equal(outs[0][1][0], outs[1][1][0]) and np.array_equal(outs[0][1][1], outs[1][1][1])


# Without streaming, the update and the products of the next step walk the slabs, a CTA each while one wave of CTAs
# covers them (1,216 on a GB300), else a warp each: 489 and 1,368 slabs of 1,024 columns; the first slab's region
# takes several passes of a warp, the last, ragged one has runs of up to 14 rows.
@pytest.mark.parametrize("residency", ["device", "host"])
@pytest.mark.parametrize("d", [500001, 1400001])
def test_updates_walk_the_slabs_one_by_one(d, residency):
    N, B, tau, lr, l2 = 8, 32, 3, 0.4, 0.02
    sh = inputs.sparse_custom(seed=11, N=N, d=d, rows=7 * B, lengths=[np.full(7 * B, 30)] * N)
    rng = np.random.default_rng(4)
    for i in range(N):
        sh.col[i][sh.rowptr[i][1:] - 1] = np.where(rng.random(7 * B) < 0.3, d - 1, sh.col[i][sh.rowptr[i][1:] - 1])
        sh.col[i][sh.rowptr[i][:-1]] = rng.integers(0, 24, 7 * B)         # 24 columns, one or two rows each
        sh.col[i][sh.rowptr[i][:-1] + 1] = rng.integers(24, 1000, 7 * B)
    W0 = (0.1 * rng.standard_normal((N, d))).astype(np.float32)
    with _make(sh, N, 1, "ring", "logistic", B, lr, l2=l2, tau=tau, residency=residency) as ctx:
        layout = ctx.debug_shard_layout()
        assert layout["entries"] and not layout["streams"]
        before = ctx.kernel_launches()
        _check(ctx, sh, 2, B, "logistic", lr, rounds.graph_schedule("ring", N, 1, graph_seed=7), l2=l2, tau=tau, W0=W0)
        # a gather at the start; per round tau steps, tau - 1 updates and gathers, a reduce
        assert ctx.kernel_launches() - before == 1 + 2 * (3 * tau - 1)


# With many workers and few entries a slab (less than two for five workers) the column lists are taken, from 257
# workers at any size, from 65 where W is more than 80 MB: either side of each line
@pytest.mark.parametrize("N,d,B,row_len,entries", [(300, 3000, 16, 4, False), (300, 3000, 16, 5, True),
                                                   (256, 3000, 8, 2, True), (65, 330000, 16, 150, True),
                                                   (65, 330000, 16, 100, False), (65, 320000, 16, 100, True),
                                                   (64, 340000, 8, 2, True)])
def test_few_entries_of_many_workers(N, d, B, row_len, entries):
    sh = inputs.sparse_custom(seed=N, N=N, d=d, rows=2 * B, lengths=[np.full(2 * B, row_len)] * N)
    with _make(sh, N, 1, "ring", "logistic", B, 0.4, tau=2) as ctx:
        assert _uses_entries(ctx) == entries
        _check(ctx, sh, 1, B, "logistic", 0.4, rounds.graph_schedule("ring", N, 1), tau=2)


# A hot column: the entries of a slab's long runs times the longest run, at most 6,000 (1,500 where there are more slabs
# than one wave of CTAs walks), else the column lists
@pytest.mark.parametrize("N,d,hot_rows,entries", [(5, 4000, 32, True), (6, 4000, 32, False), (22, 30000, 16, True),
                                                  (24, 30000, 16, False), (5, 1400000, 16, True),
                                                  (6, 1400000, 16, False), (24, 1400000, 3, True)])
def test_hot_columns(N, d, hot_rows, entries):
    B = 64
    sh = inputs.sparse_custom(seed=N, N=N, d=d, rows=2 * B, lengths=[np.full(2 * B, 6)] * N)
    for i in range(N):
        first = sh.rowptr[i][:-1]
        sh.col[i][first] = np.where(np.arange(2 * B) % B < hot_rows, 0, np.maximum(sh.col[i][first], 1))
    with _make(sh, N, 1, "ring", "logistic", B, 0.4, tau=2) as ctx:
        assert _uses_entries(ctx) == entries
        _check(ctx, sh, 2, B, "logistic", 0.4, rounds.graph_schedule("ring", N, 1), tau=2)


# Slab widths of small problems: entries in slabs as wide as half the SMs allow; entries that fit 704 a region only in
# narrower ones; column lists narrowed for their length, in two steps
@pytest.mark.parametrize("N,d,B,row_len,hot,entries", [(12, 30000, 32, 10, False, True), (5, 100000, 64, 250, False, True),
                                                       (16, 30000, 64, 300, True, False), (2, 9000, 40, 20, True, False)])
def test_slab_widths_of_small_problems(N, d, B, row_len, hot, entries):
    sh = inputs.sparse_custom(seed=B, N=N, d=d, rows=3 * B, lengths=[np.full(3 * B, row_len)] * N,
                              **({"hot_col": 7} if hot else {}))
    W0 = (0.1 * np.random.default_rng(5).standard_normal((N, d))).astype(np.float32)
    with _make(sh, N, 1, "ring", "logistic", B, 0.3, l2=0.01, tau=2) as ctx:
        assert _uses_entries(ctx) == entries
        _check(ctx, sh, 2, B, "logistic", 0.3, rounds.graph_schedule("ring", N, 1), l2=0.01, tau=2, W0=W0)
