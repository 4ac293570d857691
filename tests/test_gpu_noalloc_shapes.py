"""asap_mix_noalloc over its range (GPU): every number of inputs per row its
kernel is built for and the general one, slabs from 32 to 1,024 columns,
leading dimensions from 4 up, tables that are not doubly stochastic, against
the oracle's reduce and ||W_out - 1 wbar^T||_F with wbar the column mean of the
input.  Tolerances: 1e-6 per worker for at most 32 fp32 multiply-adds of
values of like size (32 x 2^-24 = 2e-6 at worst, a few 2^-24 in practice), 1e-5
for the error norm."""
import ctypes as C

import numpy as np
import pytest

from parity import rel_err_rows

pytestmark = pytest.mark.gpu


def _run(W, d, nbr, wgt, calls=1, drop_slab=None):
    import torch

    from paper_1612_08608_gb300._lib import load_library
    lib = load_library()
    N, ld = W.shape
    W_in, W_out = torch.from_numpy(W).cuda(), torch.full((N, ld), float("nan"), device="cuda")
    n, w = torch.from_numpy(nbr.astype(np.int32)).cuda(), torch.from_numpy(wgt.astype(np.float32)).cuda()
    cons = torch.empty(1, device="cuda")
    p = C.c_void_p
    args = (p(W_in.data_ptr()), p(W_out.data_ptr()), N, d, ld, p(n.data_ptr()), p(w.data_ptr()), nbr.shape[1],
            p(cons.data_ptr()), p(torch.cuda.current_stream().cuda_stream))
    for _ in range(calls):
        if drop_slab is None:
            st = lib.asap_mix_noalloc(*args)
        else:
            st = lib.asap_debug_mix_noalloc(*args, 20_000_000, drop_slab)
        assert st == 0, lib.asap_last_error(None)
    torch.cuda.synchronize()
    return W_out.cpu().numpy(), cons.item()


@pytest.mark.parametrize("N,ld", [(1, 4), (1, 4100), (2, 20), (3, 36), (7, 9732), (8, 4096), (9, 500000), (33, 1028),
                                  (100, 30004), (255, 644), (256, 40000)])
@pytest.mark.parametrize("kp1", [1, 2, 3, 5, 7, 32])
def test_matches_the_reduce(N, ld, kp1):
    rng = np.random.default_rng(N * 100 + kp1)
    W = rng.standard_normal((N, ld)).astype(np.float32) + 3.0 * rng.standard_normal(ld).astype(np.float32)
    nbr = rng.integers(0, N, (N, kp1))              # repeated ids and rows without the worker itself are allowed
    wgt = rng.random((N, kp1)).astype(np.float32)
    wgt /= wgt.sum(axis=1, keepdims=True)
    got, cons = _run(W, ld, nbr, wgt, calls=2)
    want = np.einsum("im,imc->ic", wgt.astype(np.float64), W.astype(np.float64)[nbr]) if N * ld * kp1 < 4e6 else \
        sum(wgt[:, m:m + 1].astype(np.float64) * W.astype(np.float64)[nbr[:, m]] for m in range(kp1))
    assert rel_err_rows(got, want) <= 1e-6
    err = np.sqrt(((want - W.astype(np.float64).mean(axis=0)) ** 2).sum())
    # the norm is off by at most the norm of the elements' errors: kp1 roundings of the output and about two of
    # the mean, each at most 2^-24 of values no larger than W's (rms)
    assert abs(cons - err) <= 1e-5 * err + (kp1 + 2) * 2.0 ** -24 * np.linalg.norm(W), (cons, err)


def test_ids_outside_the_range_are_clamped():
    W = np.arange(4 * 64, dtype=np.float32).reshape(4, 64)
    got, _ = _run(W, 64, np.array([[-5], [4], [100], [1]]), np.ones((4, 1)))
    assert np.array_equal(got, W[[0, 3, 3, 1]])


def test_calls_of_different_sizes_in_turn():
    # more calls than the scratch has slots, of one to many CTAs
    rng = np.random.default_rng(1)
    sizes = [(3, 36), (8, 4096), (64, 9000), (1, 4), (200, 700)]
    for t in range(40):
        N, ld = sizes[t % len(sizes)]
        W = rng.standard_normal((N, ld)).astype(np.float32)
        nbr = np.stack([np.arange(N), (np.arange(N) + 1) % N], axis=1)
        got, cons = _run(W, ld, nbr, np.full((N, 2), 0.5))
        want = 0.5 * (W.astype(np.float64) + W.astype(np.float64)[nbr[:, 1]])
        err = np.sqrt(((want - W.astype(np.float64).mean(axis=0)) ** 2).sum())
        assert rel_err_rows(got, want) <= 1e-6
        assert abs(cons - err) <= 1e-5 * err + 4 * 2.0 ** -24 * np.linalg.norm(W), (t, cons, err)


# N = 24 and ld = 200,000 in slabs of 256 columns: 782 slabs, five or six for each of 152 CTAs (two groups on alternate
# slabs, four stages); the slab that never lands is a CTA's first, one of the second group's, one that reuses a
# stage, and the last
@pytest.mark.parametrize("drop", [0, 152 + 7, 4 * 152 + 3, 781])
def test_a_wait_that_runs_out_makes_the_consensus_error_nan(drop):
    rng = np.random.default_rng(drop)
    N, ld, S = 24, 200000, 256
    W = rng.standard_normal((N, ld)).astype(np.float32)
    nbr = np.stack([np.arange(N), (np.arange(N) + 1) % N], axis=1)
    wgt = np.full((N, 2), 0.5)
    want = 0.5 * (W.astype(np.float64) + W.astype(np.float64)[nbr[:, 1]])
    got, cons = _run(W, ld, nbr, wgt, drop_slab=drop)
    assert np.isnan(cons)
    assert np.isnan(got[:, drop * S:(drop + 1) * S]).all()          # not written
    # slabs of the other CTAs are there
    other = [s for s in range(ld // S) if s % 152 != drop % 152]
    for s in other[::50]:
        assert rel_err_rows(got[:, s * S:(s + 1) * S], want[:, s * S:(s + 1) * S]) <= 1e-6
    # the debug entry without a dropped slab, and the next calls, are whole
    for d in (-1, None):
        got, cons = _run(W, ld, nbr, wgt, drop_slab=d)
        err = np.sqrt(((want - W.astype(np.float64).mean(axis=0)) ** 2).sum())
        assert rel_err_rows(got, want) <= 1e-6 and abs(cons - err) <= 1e-5 * err
