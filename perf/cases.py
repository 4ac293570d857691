"""Cases that measure what a user of this framework has it do, through its public entry points.

Kinds of case:
  sparse   T rounds (SGD step of every worker on its own CSR shard, then the stochastic reduce) of a
           hinge or logistic model, then the parameters and the rounds' metrics are read back;
  dense    the same with softmax regression on bf16 features;
  mix      parameters that already live in HBM are handed over, mixed T times (the reduce alone) and
           read back with the consensus errors;
  noalloc  one call of asap_mix_noalloc on tensors the caller owns.

Parameters are read into a pinned host buffer that the program keeps.  Training state moves on from pass
to pass, as a training loop's does; mix and noalloc start from the same inputs each time.
``exact`` restates every path in 64 bits with plain torch (graphs included)."""
import ctypes
import math

import numpy as np
import torch

from paper_1612_08608_gb300 import Context, inputs, load_library

GOLDEN = 0x9E3779B97F4A7C15
MASK = (1 << 64) - 1


def listed():
    return [
        # The smallest job: four workers, dense rows stored as CSR, ring with weights 1/2, 1/4, 1/4, ten
        # rounds.  Latency of the kernels and launches is all there is.
        dict(name="tiny logistic", kind="sparse", data="tiny", N=4, d=64, B=32, nnz=64, nb=8, loss="logistic", lr=0.1,
             graph="half_quarter", k=2, regen=False, T=10, tau=1, l2=0.0, gamma=0.0, sync="bsp", residency="device",
             w0=0.0),
        # Linear SVM on tf-idf text (RCV1's shape): skewed columns, ragged rows, a model that fits L2.
        dict(name="rcv1 hinge", kind="sparse", data="zipf", N=16, d=47236, B=256, nnz=75, nb=4, loss="hinge", lr=0.1,
             graph="random_regular", k=2, regen=False, T=50, tau=1, l2=0.0, gamma=0.0, sync="bsp", residency="device",
             w0=0.0),
        # The same data resumed from a checkpoint, with the options of a production run: NOTIFY-ACK, two
        # local steps per round, a decreasing rate and L2.
        dict(name="rcv1 notify-ack local steps", kind="sparse", data="zipf", N=16, d=47236, B=256, nnz=75, nb=4,
             loss="hinge", lr=0.5, graph="random_regular", k=2, regen=True, T=25, tau=2, l2=1e-4, gamma=0.01,
             sync="notify_ack", residency="device", w0=1.0),
        # Hashed features at scale (the benchmark's workload): a model larger than L2, a new graph per round.
        dict(name="hashed logistic", kind="sparse", data="uniform", N=64, d=1 << 20, B=512, nnz=100, nb=4,
             loss="logistic", lr=0.1, graph="random_regular", k=4, regen=True, T=100, tau=1, l2=0.0, gamma=0.0,
             sync="bsp", residency="device", w0=0.0),
        # The same with shards that do not fit HBM: each round's minibatch comes from pinned host memory.
        dict(name="hashed host-resident", kind="sparse", data="uniform", N=64, d=1 << 20, B=512, nnz=100, nb=4,
             loss="logistic", lr=0.1, graph="random_regular", k=4, regen=True, T=50, tau=1, l2=0.0, gamma=0.0,
             sync="bsp", residency="host", w0=0.0),
        # The same with four local steps per exchange, a decreasing rate and L2.
        dict(name="hashed local steps", kind="sparse", data="uniform", N=64, d=1 << 20, B=512, nnz=100, nb=4,
             loss="logistic", lr=0.1, graph="random_regular", k=4, regen=True, T=25, tau=4, l2=1e-4, gamma=0.001,
             sync="bsp", residency="device", w0=0.01),
        # Gossip averaging of a few small replicas: the model fits L2, latency counts.
        dict(name="mix small ring", kind="mix", N=8, d=100000, graph="ring", k=1, regen=False, T=20),
        # Gossip averaging of many replicas, larger than L2, a new graph per round.
        dict(name="mix many replicas", kind="mix", N=256, d=1000000, graph="random_regular", k=4, regen=True, T=50),
        # One reduce of tensors that a host framework owns: a small call, and a large one.
        dict(name="noalloc small", kind="noalloc", N=8, d=4093, graph="ring", k=1),
        dict(name="noalloc large", kind="noalloc", N=32, d=4000000, graph="random_regular", k=2),
        # Softmax regression on bf16 features: a small model, and the full-size one.
        dict(name="dense small", kind="dense", N=4, d=256, C=10, B=128, nb=2, lr=0.5, graph="ring", k=1, T=20, l2=0.0,
             w0=0.0),
        dict(name="dense softmax", kind="dense", N=32, d=2048, C=1000, B=512, nb=2, lr=0.1, graph="root", k=2, T=50,
             l2=0.0, w0=0.01),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph_of(rng, N, ks=(1, 2, 2, 3, 4, 4, "all")):
    k = rng.choice(ks)
    if k == "all" or k >= N - 1:
        return "complete", N - 1
    if k == 1:
        return "ring", 1
    if k == 2 and N >= 6 and rng.random() < 0.3:
        return "root", 2
    return "random_regular", k


def draw(rng):
    kind = rng.choice(["sparse", "sparse", "sparse", "mix", "noalloc", "dense"])
    if kind == "sparse":
        data = rng.choice(["uniform", "uniform", "ragged", "zipf"])
        N = _log(rng, 4, 80)
        d = _log(rng, 2000, min(1 << 20, (64 << 20) // N)) if data != "zipf" else _log(rng, 5000, 100000)
        B = _log(rng, 16, 700)
        top = min(120, int(math.sqrt(d)), 3000000 // (N * B)) if data != "zipf" else min(100, 1000000 // (N * B))
        nnz = _log(rng, 4, max(5, top))
        graph, k = _graph_of(rng, N)
        loss = rng.choice(["hinge", "logistic"])
        # hinge from a model already in training: at the corner y m = 1 rounding picks the subgradient, which
        # would show in a model that is only a few such steps old
        w0 = rng.choice([0.0, 0.1, 1.0]) if loss == "logistic" else 1.0
        return dict(kind="sparse", data=data, N=N, d=d, B=B, nnz=nnz, nb=rng.choice([2, 3, 4]),
                    loss=loss, lr=rng.choice([0.1, 0.3, 0.5]), graph=graph, k=k,
                    regen=graph == "random_regular" and rng.random() < 0.5, T=rng.choice([10, 20, 30]),
                    tau=rng.choice([1, 1, 2, 3]), l2=rng.choice([0.0, 1e-4]), gamma=rng.choice([0.0, 0.01]),
                    sync=rng.choice(["bsp", "bsp", "notify_ack"]), residency=rng.choice(["device", "device", "host"]), w0=w0)
    if kind == "mix":
        N = _log(rng, 2, 256)
        d = _log(rng, 1000, (250 << 20) // N) if N > 25 else _log(rng, 1000, 10000000)
        graph, k = _graph_of(rng, N)
        return dict(kind="mix", N=N, d=d, graph=graph, k=k, regen=graph == "random_regular" and rng.random() < 0.5,
                    T=rng.choice([10, 20, 40]))
    if kind == "noalloc":
        N = _log(rng, 2, 256)
        S = 256
        while S > 4 and N * S * 4 > 16384:
            S //= 2
        d = _log(rng, 1000, min(128000000 // N, 32768 * S))
        graph, k = _graph_of(rng, N, (1, 2, 3, 4, 6))
        if k > 31:
            graph, k = "ring", 1
        return dict(kind="noalloc", N=N, d=d, graph=graph, k=k)
    N, B, C = _log(rng, 2, 32), 128 * rng.choice([1, 2, 3, 4]), _log(rng, 2, 1000)
    d = 256 * _log(rng, 1, 8)
    graph, k = _graph_of(rng, N)
    return dict(kind="dense", N=N, d=d, C=C, B=B, nb=2, lr=rng.choice([0.1, 0.5]), graph=graph, k=k,
                T=rng.choice([10, 20]), l2=rng.choice([0.0, 0.01]), w0=rng.choice([0.0, 0.01]))


# ---- inputs ---------------------------------------------------------------------------------------------
def _shards(case, seed):
    N, d, rows, nnz = case["N"], case["d"], case["nb"] * case["B"], case["nnz"]
    if case["data"] == "tiny":
        return inputs.tiny_dense_logistic(seed=seed, N=N, d=d, rows=rows)
    if case["data"] == "zipf":
        return inputs.sparse_hinge_svm(seed=seed, N=N, d=d, rows=rows, mean_nnz=float(nnz))
    if case["data"] == "uniform":
        return inputs.sparse_logistic_hashed(seed=seed, N=N, d=d, rows=rows, nnz=nnz)
    return inputs.sparse_custom(seed=seed, N=N, d=d, rows=rows, max_len=2 * nnz)   # ragged, empty rows too


def _randn(shape, seed, dtype=torch.float32):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _dense_inputs(case, seed):
    """bf16 features [N, rows, d] and the labels argmax(x W*^T + Gumbel) [N, rows]."""
    N, d, C, rows = case["N"], case["d"], case["C"], case["nb"] * case["B"]
    X = _randn((N, rows, d), seed).to(torch.bfloat16)
    teacher = (_randn((C, d), seed + 1) / math.sqrt(d)).to(torch.bfloat16)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 19)
    y = torch.empty((N, rows), dtype=torch.int64, device="cuda")
    for i in range(N):
        u = torch.rand((rows, C), generator=g, device="cuda").clamp_(1e-20, 1.0 - 1e-7)
        y[i] = ((X[i] @ teacher.T).float() - torch.log(-torch.log(u))).argmax(dim=1)
    return X, y


def _pinned(N, P):
    return torch.empty((N, P), dtype=torch.float32, pin_memory=True)


def _start(case, seed, P):
    return case["w0"] * _randn((case["N"], P), seed + 3)


def _set_graph(ctx, case):
    if case["graph"] == "half_quarter":
        ctx.set_mixing(*_half_quarter(case["N"]))
    else:
        ctx.set_graph(case["graph"], regenerate=bool(case.get("regen", False)))


def prepare(case, seed):
    kind, N, d = case["kind"], case["N"], case["d"]
    if kind == "noalloc":
        ld = (d + 3) // 4 * 4
        W = torch.zeros((N, ld), dtype=torch.float32, device="cuda")
        W[:, :d] = _randn((N, d), seed)
        nbr, wgt = _graph(case["graph"], N, case["k"], 5, 0)
        return dict(kind=kind, N=N, d=d, ld=ld, kp1=nbr.shape[1], W=W, out=torch.empty_like(W),
                    nbr=torch.from_numpy(nbr.astype(np.int32)).cuda(),
                    wgt=torch.from_numpy(wgt.astype(np.float32)).cuda(),
                    cons=torch.empty(1, dtype=torch.float32, device="cuda"), lib=load_library())
    ctx = Context(N, d, graph_seed=5, k=case["k"])
    s = dict(kind=kind, ctx=ctx, T=case["T"])
    if kind == "mix":
        _set_graph(ctx, case)
        s["W0"], s["out"] = _randn((N, d), seed), _pinned(N, d)
        return s
    if kind == "sparse":
        ctx.set_model(case["loss"], batch=case["B"], lr=case["lr"], l2=case["l2"])
        _set_graph(ctx, case)
        ctx.set_schedule(case["tau"], "inverse" if case["gamma"] else "constant", case["gamma"])
        ctx.set_shard_residency(case["residency"])
        ctx.set_sync_mode(case["sync"])
        ctx.load_shards(_shards(case, seed))
        P = d
    else:
        ctx.set_model("softmax", batch=case["B"], lr=case["lr"], num_classes=case["C"], l2=case["l2"])
        _set_graph(ctx, case)
        X, y = _dense_inputs(case, seed)
        bits, ids = X.view(torch.int16).cpu().numpy().view(np.uint16), y.to(torch.int32).cpu().numpy()
        ctx.load_dense_shards(X=list(bits), y=list(ids))
        P = d * case["C"]
    if case["w0"]:
        W0 = _start(case, seed, P)
        torch.cuda.synchronize()                       # drawn on torch's stream, copied on the context's
        ctx.write_params_device(W0, 0)
    s["out"] = _pinned(N, P)
    return s


def run(s):
    if s["kind"] == "noalloc":
        p = ctypes.c_void_p
        status = s["lib"].asap_mix_noalloc(p(s["W"].data_ptr()), p(s["out"].data_ptr()), s["N"], s["d"], s["ld"],
                                           p(s["nbr"].data_ptr()), p(s["wgt"].data_ptr()), s["kp1"],
                                           p(s["cons"].data_ptr()), p(torch.cuda.current_stream().cuda_stream))
        if status != 0:
            raise RuntimeError("asap_mix_noalloc: status %d" % status)
        return s["out"], s["cons"]
    ctx, T = s["ctx"], s["T"]
    if s["kind"] == "mix":
        ctx.write_params_device(s["W0"], 0)
    ctx.round(T)
    _, rnd = ctx.read_params(s["out"].numpy())
    loss, cons = ctx.read_metrics(rnd - T, T)
    return (s["out"], cons) if s["kind"] == "mix" else (s["out"], loss, cons)


# ---- what a pass cannot do without ------------------------------------------------------------------------
def work(case):
    N, d, kp1 = case["N"], case["d"], case["k"] + 1
    if case["kind"] == "noalloc":
        return dict(bytes=8.0 * N * d, flops=2.0 * kp1 * N * d)
    T = case["T"]
    mix = 2.0 * kp1 * N * d if case["graph"] != "complete" else 2.0 * N * d
    if case["kind"] == "mix":
        return dict(bytes=(8.0 * T + 4.0) * N * d, flops=T * mix)
    if case["kind"] == "sparse":
        # per local step: column id and value of every entry once, one label per row; a step whose update is
        # not folded into the reduce reads and writes the parameters its entries touch
        E = float(N * case["B"] * case["nnz"])
        step = 8.0 * E + 4.0 * N * case["B"]
        return dict(bytes=T * (8.0 * N * d + case["tau"] * step + (case["tau"] - 1) * 8.0 * E) + 4.0 * N * d,
                    flops=T * (mix + case["tau"] * 4.0 * E))
    # forward and gradient GEMM; parameters read and written by the update and by the reduce
    C, B = case["C"], case["B"]
    return dict(bytes=T * (16.0 * N * C * d + 2.0 * N * B * d) + 4.0 * N * C * d,
                flops=T * (4.0 * N * B * C * d + 2.0 * kp1 * N * C * d))


def tolerance(case):
    # About four times the distance from exact() as measured: 5e-4 for bf16 operands over up to 50 rounds,
    # up to 1e-6 for 32-bit sums carried over many rounds, 7e-8 for a single reduce.
    if case["kind"] == "dense":
        return {"rel": 2e-3}
    return {"rel": 5e-7} if case["kind"] == "noalloc" else {"rel": 4e-6}


# ---- the same in 64 bits, in plain torch ------------------------------------------------------------------
class _SplitMix64:
    def __init__(self, state):
        self.s = state & MASK

    def below(self, m):
        limit = (1 << 64) - ((1 << 64) % m)
        while True:
            self.s = (self.s + GOLDEN) & MASK
            z = self.s
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & MASK
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK
            z ^= z >> 31
            if z < limit:
                return z % m


def _half_quarter(N):
    rows = [sorted([((i - 1) % N, 0.25), (i, 0.5), ((i + 1) % N, 0.25)]) for i in range(N)]
    return (np.array([[j for j, _ in r] for r in rows], np.int32),
            np.array([[w for _, w in r] for r in rows], np.float32))


def _graph(kind, N, k, seed, rnd):
    """In-neighbours (the worker itself among them, ascending) and weights of every worker."""
    if kind == "half_quarter":
        return _half_quarter(N)
    if kind == "ring":
        sets = [{i, (i - 1) % N} for i in range(N)]
    elif kind == "root":
        sets = [{i, (i - 1) % N, (i - math.isqrt(N)) % N} for i in range(N)]
    elif kind == "complete":
        sets = [set(range(N)) for _ in range(N)]
    else:
        rng = _SplitMix64(seed ^ ((GOLDEN * (rnd + 1)) & MASK))
        pi = list(range(N))
        for t in range(N - 1, 0, -1):
            j = rng.below(t + 1)
            pi[t], pi[j] = pi[j], pi[t]
        sets = [set() for _ in range(N)]
        for t in range(N):
            sets[pi[(t + 1) % N]].add(pi[t])
        for _ in range(k - 1):
            while True:
                sigma, good = list(range(N)), True
                for t in range(N - 1, -1, -1):
                    if t:
                        j = rng.below(t + 1)
                        sigma[t], sigma[j] = sigma[j], sigma[t]
                    if sigma[t] == t or sigma[t] in sets[t]:
                        good = False
                        break
                if good:
                    break
            for i in range(N):
                sets[i].add(sigma[i])
        for i in range(N):
            sets[i].add(i)
    nbr = np.array([sorted(s) for s in sets], np.int64)
    return nbr, np.full(nbr.shape, 1.0 / nbr.shape[1])


def _mix(W, case, rnd):
    if case["graph"] == "complete":
        return W.mean(dim=0, keepdim=True).expand_as(W).clone()
    nbr, wgt = _graph(case["graph"], case["N"], case["k"], 5, rnd if case.get("regen") else 0)
    nbr, wgt = torch.from_numpy(nbr.astype(np.int64)).cuda(), torch.from_numpy(wgt.astype(np.float64)).cuda()
    out = torch.zeros_like(W)
    for m in range(nbr.shape[1]):
        out += wgt[:, m:m + 1] * W[nbr[:, m]]
    return out


def _consensus(W):
    return float((W - W.mean(dim=0)).square().sum().sqrt())


def exact(case, seed):
    kind, N, d = case["kind"], case["N"], case["d"]
    if kind == "noalloc":
        ld = (d + 3) // 4 * 4
        W = torch.zeros((N, ld), dtype=torch.float64, device="cuda")
        W[:, :d] = _randn((N, d), seed).double()
        out = _mix(W, case, 0)
        return out, torch.tensor([float((out - W.mean(dim=0)).square().sum().sqrt())], dtype=torch.float64)
    if kind == "mix":
        W, cons = _randn((N, d), seed).double(), []
        for t in range(case["T"]):
            W = _mix(W, case, t)
            cons.append(_consensus(W))
        return W, np.array(cons)
    return _exact_sparse(case, seed) if kind == "sparse" else _exact_dense(case, seed)


def _exact_sparse(case, seed):
    N, d, B, nb = case["N"], case["d"], case["B"], case["nb"]
    sh = _shards(case, seed)
    batches = []                                       # per minibatch: flat parameter index, row, value, label
    for t in range(nb):
        idx, row, val, y = [], [], [], []
        for i in range(N):
            rp = sh.rowptr[i][t * B:(t + 1) * B + 1]
            idx.append(sh.col[i][rp[0]:rp[-1]].astype(np.int64) + i * d)
            row.append(np.repeat(np.arange(B), np.diff(rp)) + i * B)
            val.append(sh.val[i][rp[0]:rp[-1]].astype(np.float64))
            y.append(sh.y[i][t * B:(t + 1) * B].astype(np.float64))
        batches.append([torch.from_numpy(np.concatenate(v)).cuda() for v in (idx, row, val, y)])
    W = _start(case, seed, d).double()
    losses, cons = [], []
    for t in range(case["T"]):
        for j in range(case["tau"]):
            k = t * case["tau"] + j
            idx, row, val, y = batches[k % nb]
            eta = case["lr"] / (1.0 + case["gamma"] * k)
            m = torch.zeros(N * B, dtype=torch.float64, device="cuda").index_add_(0, row, val * W.view(-1)[idx])
            z = y * m
            if case["loss"] == "hinge":
                loss, r = (1.0 - z).clamp(min=0.0), torch.where(z < 1.0, -y, torch.zeros_like(y))
            else:
                loss, r = torch.nn.functional.softplus(-z), -y * torch.sigmoid(-z)
            W = W * (1.0 - eta * case["l2"])
            W.view(-1).index_add_(0, idx, (-eta / B) * r[row] * val)
        losses.append(float(loss.mean()))
        W = _mix(W, case, t)
        cons.append(_consensus(W))
    return W, np.array(losses), np.array(cons)


def _exact_dense(case, seed):
    N, d, C, B, nb, eta = case["N"], case["d"], case["C"], case["B"], case["nb"], case["lr"]
    X, y = _dense_inputs(case, seed)
    W = _start(case, seed, C * d).double()
    losses, cons = [], []
    for t in range(case["T"]):
        b = slice((t % nb) * B, (t % nb) * B + B)
        Xb, yb = X[:, b].double(), y[:, b]
        Wm = W.view(N, C, d)
        Z = torch.bmm(Xb, Wm.transpose(1, 2))
        losses.append(float((torch.logsumexp(Z, dim=2) - Z.gather(2, yb[:, :, None])[:, :, 0]).mean()))
        R = torch.softmax(Z, dim=2)
        R.scatter_add_(2, yb[:, :, None], torch.full((N, B, 1), -1.0, dtype=torch.float64, device="cuda"))
        W = ((1.0 - eta * case["l2"]) * Wm - (eta / B) * torch.bmm(R.transpose(1, 2), Xb)).reshape(N, C * d)
        W = _mix(W, case, t)
        cons.append(_consensus(W))
    return W, np.array(losses), np.array(cons)
