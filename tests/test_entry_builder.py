"""The library's builder of the entry layout (host only, no GPU): the image that
asap_load_shards uploads for evenly spread columns, decoded and checked
against a plain restatement from the shards -- labels and entry counts, per
slab the entries by (worker, column, row) with their run flags, values and
places, the padding, and no run across a multiple of 32 entries of its region."""
import numpy as np
import pytest

from paper_1612_08608_gb300 import inputs
from paper_1612_08608_gb300.api import AsapError, debug_entry_image

PAD, OFF, MORE, NEXT = 0xFFFFFFFF, 0x3FFF, 0x4000, 0x8000


def _view(img, off, dtype, n):
    return np.frombuffer(img[off:off + np.dtype(dtype).itemsize * n].tobytes(), dtype=dtype)


def _check_image(sh, B, S, t):
    N, d = sh.N, sh.d
    img, o = debug_entry_image(sh, B, S, t)
    n_slabs = -(-((d + 63) // 64 * 64) // S)
    soff = _view(img, o["soff"], np.int32, n_slabs + 1)
    assert soff[0] == 0 and np.all(np.diff(soff) >= 0) and np.all(soff % 8 == 0)
    assert o["max_region"] == np.diff(soff).max(initial=0)
    code = _view(img, o["code"], np.uint32, soff[-1])
    val = _view(img, o["val"], np.float32, soff[-1])
    packed = o["place"] < 0
    longest = max(int(np.diff(sh.rowptr[i][t * B:(t + 1) * B + 1]).max()) for i in range(N))
    bits = lambda n: max(1, int(n - 1).bit_length()) if n > 1 else 0
    assert packed == (max(1, bits(longest)) + bits(B) <= 16) and o["row_shift"] == 16 + packed * max(1, bits(longest))
    assert all(o[k] % 16 == 0 for k in ("y", "len", "soff", "code", "val")) and (packed or o["place"] % 16 == 0)

    want = {s: [] for s in range(n_slabs)}
    for i in range(N):
        r0 = t * B
        assert np.array_equal(_view(img, o["y"], np.float32, N * B)[i * B:(i + 1) * B], sh.y[i][r0:r0 + B])
        assert np.array_equal(_view(img, o["len"], np.uint16, N * B)[i * B:(i + 1) * B],
                              np.diff(sh.rowptr[i][r0:r0 + B + 1]))
        for b in range(B):
            a, e = sh.rowptr[i][r0 + b], sh.rowptr[i][r0 + b + 1]
            for j in range(e - a):
                c = int(sh.col[i][a + j])
                want[c // S].append((i, c % S, b, j, sh.val[i][a + j]))
    longest_run = 0
    for s in range(n_slabs):
        got = []
        rc = code[soff[s]:soff[s + 1]]
        for e, c in enumerate(int(x) for x in rc):
            if c == PAD:
                assert val[soff[s] + e] == 0.0
                continue
            off = c & OFF
            if packed:
                place = (c >> 16) & ((1 << (o["row_shift"] - 16)) - 1)
            else:
                place = int(_view(img, o["place"], np.uint16, soff[-1])[soff[s] + e])
            got.append((off // S, off % S, c >> o["row_shift"], place, val[soff[s] + e], e, c))
        assert [g[:5] for g in got] == sorted(want[s], key=lambda x: x[:3])
        # runs of one (worker, column): flagged, without padding inside, in one group of 32
        k = 0
        while k < len(got):
            run = [g for g in got[k:k + 64] if g[:2] == got[k][:2]]
            longest_run = max(longest_run, len(run))
            assert [g[5] for g in run] == list(range(run[0][5], run[0][5] + len(run)))
            assert run[0][5] // 32 == run[-1][5] // 32
            assert [bool(g[6] & NEXT) for g in run] == [False] + [True] * (len(run) - 1)
            assert [bool(g[6] & MORE) for g in run] == [True] * (len(run) - 1) + [False]
            k += len(run)
    assert o["max_run"] == longest_run
    return o


@pytest.mark.parametrize("S,max_len,packed", [(8, 12, True), (64, 40, True), (1024, 40, True), (32, 900, False)])
def test_image_matches_the_shards(S, max_len, packed):
    N, d, B = 3, 1000, 100 if not packed else 20
    rng = np.random.default_rng(S)
    lengths = [np.where(rng.random(3 * B) < 0.15, 0, rng.integers(1, max_len, 3 * B)) for _ in range(N)]
    if packed:
        sh = inputs.sparse_custom(seed=31, N=N, d=d, rows=3 * B, lengths=lengths)
    else:                                 # 100 rows of up to 899 places: 7 + 10 bits; runs stay short in 40,000 columns
        d = 40000
        sh = inputs.sparse_custom(seed=31, N=N, d=d, rows=3 * B, lengths=lengths)
    for t in (0, 1, 2):
        o = _check_image(sh, B, S, t)
        assert (o["place"] < 0) == packed


def test_long_runs_empty_minibatches_and_the_edges_of_the_code():
    # worker 0: columns shared by 32, 31, 17 and 16 rows, next to each other, so that runs meet multiples of 32;
    # worker 1: nothing; worker 2: the first and the last column of every slab; worker 15: the highest code of a slab
    N, B, S = 16, 32, 512
    d = 4 * S
    rowptr, col, val, y = [], [], [], []
    rng = np.random.default_rng(0)
    for i in range(N):
        rows = []
        for b in range(B):
            c = []
            if i == 0:
                c = [k for k, n in enumerate((32, 31, 17, 16, 3, 32, 1, 30)) if b < n]
            elif i == 2:
                c = [s * S + e for s in range(4) for e in (0, S - 1) if (b + s + e) % 2 == 0]
            elif i == 15:
                c = [d - 1] if b == B - 1 else []
            rows.append(c)
        rowptr.append(np.concatenate([[0], np.cumsum([len(c) for c in rows])]).astype(np.int64))
        col.append(np.array([c for r in rows for c in r], np.int32))
        val.append(rng.standard_normal(col[-1].shape[0]).astype(np.float32))
        y.append(np.where(rng.random(B) < 0.5, -1.0, 1.0).astype(np.float32))
    sh = inputs.sparse_custom(seed=1, N=N, d=d, rows=B, max_len=4)
    sh.rowptr, sh.col, sh.val, sh.y = rowptr, col, val, y
    assert _check_image(sh, B, S, 0)["max_run"] == 32


def test_a_run_beyond_32_and_bad_columns_are_refused():
    sh = inputs.sparse_custom(seed=5, N=2, d=500, rows=64, max_len=8, hot_col=7)
    with pytest.raises(AsapError, match="too many entries"):
        debug_entry_image(sh, 64, 64, 0)
    sh = inputs.sparse_custom(seed=5, N=2, d=500, rows=64, max_len=8)
    sh.col[1][3] = 500
    with pytest.raises(AsapError, match="out of range"):
        debug_entry_image(sh, 64, 64, 0)
    with pytest.raises(AsapError):
        debug_entry_image(sh, 64, 48, 0)
