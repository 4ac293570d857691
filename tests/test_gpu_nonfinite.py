"""Parameters that are not finite (GPU): the consensus error says so, in the
context's reduce and in asap_mix_noalloc."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("N,d,k", [(4, 100, 1), (8, 70001, 3), (5, 3000, 4)])
def test_consensus_error_is_nan(bad, N, d, k):
    import torch
    from paper_1612_08608_gb300 import Context, build_graph
    from paper_1612_08608_gb300._lib import load_library
    W0 = np.random.default_rng(k).standard_normal((N, d)).astype(np.float32)
    W0[N - 1, d // 2] = bad
    kind = {1: "ring", N - 1: "complete"}.get(k, "random_regular")
    with Context(N, d, graph_seed=0, k=k) as ctx:
        ctx.set_graph(kind)
        ctx.write_params(W0, 0)
        ctx.round(1)
        cons = ctx.read_metrics(0, 1)[1][0]
        assert cons == 0.0 if kind == "complete" else np.isnan(cons)      # complete: all rows are the same
        ctx.write_params(np.zeros_like(W0), 0)
        ctx.round(1)
        assert ctx.read_metrics(0, 1)[1][0] == 0.0     # and the next round is not spoilt
    lib, ld = load_library(), (d + 3) // 4 * 4
    W_in, W_out = torch.zeros(N, ld, device="cuda"), torch.empty(N, ld, device="cuda")
    W_in[:, :d] = torch.from_numpy(W0)
    nbr = torch.from_numpy(build_graph(kind, N, k)).cuda()
    wgt = torch.full((N, k + 1), 1.0 / (k + 1), device="cuda")
    cons = torch.zeros(1, device="cuda")
    p = C.c_void_p
    assert lib.asap_mix_noalloc(p(W_in.data_ptr()), p(W_out.data_ptr()), N, d, ld, p(nbr.data_ptr()),
                                p(wgt.data_ptr()), k + 1, p(cons.data_ptr()),
                                p(torch.cuda.current_stream().cuda_stream)) == 0
    assert np.isnan(cons.item())
