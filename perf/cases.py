"""What the framework is measured on: the calls that a user's program makes, at the sizes of
this repository's own workloads and over the ranges around them.

A case is a dict of plain values; its "path" names the family:

  ragged_row  marshal a list of sequences, fused map + segmented sum, max, and a loop
  segreduce   fused map + segmented reduce of flat data
  marshal     flatten a list of separately stored sequences
  patterns    map, map2, reduce and loop over flat arrays
  fp32        per-sequence log-likelihoods, FP32 log space
  bf16        per-sequence log-likelihoods, BF16 tensor cores
  adjoint     gradients and log-likelihoods in one call
  train       one training iteration: autograd forward and backward, then the re-estimation
  gravity     records to arrays, then the all-pairs accelerations
  pairhist    all-pairs histogram of angular separations
  long        log-likelihoods of few, very long sequences
"""
import math

import numpy as np
import torch

from paper_2211_00621_gb300 import api

DEV = "cuda"
DTYPES = {"int32": torch.int32, "int64": torch.int64, "float32": torch.float32, "float64": torch.float64}
REDS = {"add": api.RED_ADD, "min": api.RED_MIN, "max": api.RED_MAX}
MAPS = {"identity": api.MAP_IDENTITY, "sq_plus_one": api.MAP_SQ_PLUS_ONE, "abs": api.MAP_ABS, "scale": api.MAP_SCALE}


def listed():
    return [
        # the smallest program: a list of 4,096 short sequences straight from the host's pointer
        # tables, one segmented sum, its maximum, and one loop -- launches and latency
        dict(name="ragged_row_4096", path="ragged_row", S=4096, hi=256),
        # the same reduction at memory scale: 2^20 ragged segments, 134M int32 elements
        dict(name="segsum_1M_segments", path="segreduce", S=1 << 20, hi=256, dtype="int32", op="add", map="sq_plus_one",
             scalar=0.0),
        # marshaling at memory scale: 2^17 separately stored pieces in shuffled places
        dict(name="marshal_131072", path="marshal", S=1 << 17, hi=256, dtype="int32"),
        # the flat patterns on a large float array: map, map2, reduce, loop (b = 2a)
        dict(name="patterns_64M", path="patterns", n=1 << 26, dtype="float32"),
        # exact-as-FP32 scoring of a small model: 512 sequences of 1,000 symbols, 64 states
        dict(name="fp32_k64", path="fp32", K=64, M=32, S=512, kind="fixed", lo=1000, hi=1000),
        # the same scoring of a large model on ragged sequences
        dict(name="fp32_k256", path="fp32", K=256, M=64, S=1024, kind="uniform", lo=200, hi=2000),
        # batched scoring on the tensor cores: 4,096 sequences of very uneven lengths
        dict(name="bf16_k256", path="bf16", K=256, M=64, S=4096, kind="loguniform", lo=50, hi=5000),
        # the gradients of the large model, forward and backward in one call
        dict(name="adjoint_k256", path="adjoint", K=256, M=64, S=1024, kind="uniform", lo=200, hi=2000),
        # a training iteration of a middle-sized model whose state count is no power of two
        dict(name="train_k100", path="train", K=100, M=40, S=200, kind="uniform", lo=20, hi=400),
        # softened gravity on 65,536 bodies handed over as records
        dict(name="gravity_65536", path="gravity", n=65536, eps=1e-3),
        # two-point correlation of 32,768 sky positions, 20 log-spaced bins
        dict(name="pairhist_32768", path="pairhist", n=32768, nb=0, bins=20),
        # scoring of four sequences of 250,000 symbols
        dict(name="long_k64", path="long", K=64, M=32, S=4, kind="fixed", lo=250000, hi=250000),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _hmm_case(rng, path, K, M, S_hi, lo, hi, sum_hi):
    kind = rng.choice(["fixed", "uniform", "loguniform"])
    S = _log_int(rng, 1 if path == "long" else 16, S_hi)
    hi = _log_int(rng, 4 * lo, hi)
    hi = max(lo, min(hi, sum_hi // S))
    return dict(path=path, K=K, M=M, S=S, kind=kind, lo=hi if kind == "fixed" else lo, hi=hi)


def draw(rng):
    path = rng.choice(["ragged_row", "segreduce", "marshal", "patterns", "fp32", "fp32", "bf16", "bf16", "adjoint",
                       "adjoint", "train", "gravity", "pairhist", "long"])
    if path == "ragged_row":
        return dict(path=path, S=_log_int(rng, 64, 8192), hi=_log_int(rng, 16, 256))
    if path == "segreduce":
        dtype = rng.choice(["int32", "int32", "int64", "float32", "float64"])
        hi = _log_int(rng, 4, 4096)
        most = (1 << 27) // (DTYPES[dtype].itemsize // 4)
        return dict(path=path, S=_log_int(rng, 1 << 10, min(1 << 20, most // hi * 2)), hi=hi, dtype=dtype,
                    op=rng.choice(["add", "add", "min", "max"]), map=rng.choice(list(MAPS)), scalar=3.0)
    if path == "marshal":
        return dict(path=path, S=_log_int(rng, 1 << 8, 1 << 17), hi=_log_int(rng, 16, 256),
                    dtype=rng.choice(["int32", "float32", "int64"]))
    if path == "patterns":
        dtype = rng.choice(["int32", "float32", "float32", "float64"])
        return dict(path=path, n=_log_int(rng, 1 << 12, 1 << (26 if dtype.endswith("32") else 25)) | 1, dtype=dtype)
    if path == "fp32":
        if rng.random() < 0.5:
            return _hmm_case(rng, path, rng.randint(2, 64), rng.randint(2, 64), 2048, 20, 2000, 512000)
        return _hmm_case(rng, path, rng.randint(65, 256), rng.randint(2, 64), 1024, 20, 2000, 1000000)
    if path == "bf16":
        return _hmm_case(rng, path, rng.choice([64, 128, 192, 256]), rng.randint(2, 64), 4096, 50, 5000, 4000000)
    if path == "adjoint":
        K = rng.choice([64, 128, 256, 256, rng.randint(5, 255)])
        return _hmm_case(rng, path, K, rng.randint(2, 64), 1024, 20, 2000, 1000000)
    if path == "train":
        return _hmm_case(rng, path, rng.choice([64, 128, rng.randint(5, 128)]), rng.randint(2, 64), 256, 5, 400, 50000)
    if path == "gravity":
        return dict(path=path, n=_log_int(rng, 100, 65536), eps=rng.choice([1e-3, 1e-2]))
    if path == "pairhist":
        n = _log_int(rng, 500, 23000)
        return dict(path=path, n=n, nb=rng.choice([0, _log_int(rng, 500, 23000)]), bins=rng.randint(5, 30))
    return _hmm_case(rng, path, rng.choice([64, 32, rng.randint(2, 64)]), rng.randint(2, 64), 8, 5000, 250000, 1000000)


# ------------------------------------------------------------------------------- inputs
def _gen(seed, k):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + k)


def _lengths(case, seed):
    """The case's lengths: the quantiles of its distribution (so that the work of a case does
    not depend on the seed), in an order drawn from the seed."""
    S = case["S"]
    u = (np.arange(S) + 0.5) / S
    lo, hi = case.get("lo", 0), case["hi"]
    kind = case.get("kind", "uniform")
    if kind == "fixed":
        x = np.full(S, hi, np.int64)
    elif kind == "loguniform":
        x = np.rint(np.exp(np.log(lo) + u * (np.log(hi) - np.log(lo)))).astype(np.int64)
    else:
        x = np.floor(lo + u * (hi + 1 - lo)).astype(np.int64)
    x = np.clip(x, lo, hi)
    return x if seed is None else np.random.default_rng(seed).permutation(x)


def _offsets(lengths):
    off = np.zeros(len(lengths) + 1, np.int64)
    np.cumsum(lengths, out=off[1:])
    return off


def _values(n, dtype, g):
    if dtype.is_floating_point:
        return torch.empty(n, dtype=dtype, device=DEV).uniform_(-1.0, 1.0, generator=g)
    return torch.randint(-1000, 1001, (n,), dtype=dtype, device=DEV, generator=g)


def _hmm(case, seed):
    K, M = case["K"], case["M"]
    g = _gen(seed, 1)

    def rows(r, c):
        e = torch.empty(r, c, dtype=torch.float64, device=DEV).exponential_(1.0, generator=g)
        return (e / e.sum(1, keepdim=True)).log().float()

    lengths = _lengths(case, seed)
    off = _offsets(lengths)
    return dict(case=case, log_A=rows(K, K), log_B=rows(K, M),
                log_pi=torch.full((K,), -math.log(K), dtype=torch.float32, device=DEV),
                obs=torch.randint(0, M, (int(off[-1]),), dtype=torch.int32, device=DEV, generator=g),
                offsets=torch.from_numpy(off).to(DEV), max_T=int(lengths.max()))


def _pieces(case, seed, dtype):
    """Separately stored sequences: views of one buffer, placed in a shuffled order."""
    lengths = _lengths(case, seed)
    place = np.random.default_rng(seed + 1).permutation(len(lengths))
    src = _values(int(lengths.sum()), dtype, _gen(seed, 2))
    stored = torch.split(src, lengths[place].tolist())
    seqs = [None] * len(lengths)
    for k, p in enumerate(place.tolist()):
        seqs[p] = stored[k]
    return seqs


def _sky(n, g):
    v = torch.empty(n, 3, dtype=torch.float64, device=DEV).normal_(generator=g)
    return (v / v.norm(dim=1, keepdim=True)).float()


def _edges(bins):
    k = np.arange(bins + 1) / bins
    return np.cos(1.0 * 10000.0 ** k * math.pi / (180 * 60)).astype(np.float32)


def prepare(case, seed):
    path = case["path"]
    if path in ("fp32", "bf16", "adjoint", "long"):
        return _hmm(case, seed)
    if path == "train":
        s = _hmm(case, seed)
        for k in ("log_A", "log_B", "log_pi"):
            s[k].requires_grad_(True)
        return s
    if path in ("ragged_row", "marshal"):
        return dict(case=case, table=api.ragged_table(_pieces(case, seed, DTYPES[case.get("dtype", "int32")])))
    if path == "segreduce":
        off = _offsets(_lengths(case, seed))
        return dict(case=case, data=_values(int(off[-1]), DTYPES[case["dtype"]], _gen(seed, 3)),
                    offsets=torch.from_numpy(off).to(DEV))
    if path == "patterns":
        return dict(case=case, x=_values(case["n"], DTYPES[case["dtype"]], _gen(seed, 4)))
    if path == "gravity":
        aos = torch.empty(case["n"], 4, dtype=torch.float32, device=DEV).uniform_(0.0, 1.0, generator=_gen(seed, 5))
        aos[:, 3] += 0.5
        return dict(case=case, aos=aos, fields=[(4 * k, torch.float32) for k in range(4)])
    g = _gen(seed, 6)
    return dict(case=case, A=_sky(case["n"], g), B=_sky(case["nb"], g) if case["nb"] else None,
                edges=torch.from_numpy(_edges(case["bins"])))


# --------------------------------------------------------------------------------- calls
def run(s):
    case = s["case"]
    path = case["path"]
    if path in ("fp32", "bf16"):
        return api.hmm_forward(s["log_A"], s["log_B"], s["log_pi"], s["obs"], s["offsets"],
                               api.HMM_FP32_LOG if path == "fp32" else api.HMM_BF16_SCALED)
    if path == "adjoint":
        return api.hmm_adjoint(s["log_A"], s["log_B"], s["log_pi"], s["obs"], s["offsets"], max_T=s["max_T"])
    if path == "long":
        return api.hmm_forward_long(s["log_A"], s["log_B"], s["log_pi"], s["obs"], s["offsets"], max_T=s["max_T"])
    if path == "train":
        p = (s["log_A"], s["log_B"], s["log_pi"])
        ll = api.HMMLogLik.apply(*p, s["obs"], s["offsets"], api.HMM_FP32_LOG, s["max_T"])
        g = torch.autograd.grad(ll.sum(), p)
        theta, new = api.hmm_mstep(*(t.detach() for t in p), *g)
        return dict(ll=ll.detach(), grad=g, theta=theta, new=new)
    if path == "ragged_row":
        flat, off = api.accel_marshal_ragged_table(s["table"])
        seg = api.accel_segreduce(api.RED_ADD, api.MAP_SQ_PLUS_ONE, flat, off, torch.int64)
        top = api.accel_reduce(api.RED_MAX, seg)
        twice = api.accel_loop(api.LOOP_SCALE, torch.empty_like(flat), flat, 2.0)
        return seg, top, twice
    if path == "marshal":
        return api.accel_marshal_ragged_table(s["table"])
    if path == "segreduce":
        return api.accel_segreduce(REDS[case["op"]], MAPS[case["map"]], s["data"], s["offsets"], scalar=case["scalar"])
    if path == "patterns":
        x = s["x"]
        wide = x.dtype if x.dtype.is_floating_point else torch.int64
        y = api.accel_map(api.MAP_SQ_PLUS_ONE, x, wide)
        z = api.accel_map(api.MAP_ADD2, x, x.dtype, y=x)
        total = api.accel_reduce(api.RED_ADD, y)
        return y, z, total, api.accel_loop(api.LOOP_SCALE, torch.empty_like(x), x, 2.0)
    if path == "gravity":
        x, y, z, m = api.accel_marshal_records(s["aos"], s["fields"])
        return api.pairwise_mapreduce(x, y, z, m, case["eps"])
    return api.accel_pair_histogram(s["A"], s["edges"], s["B"])


# ---------------------------------------------------------------------------------- work
def work(case):
    path = case["path"]
    if path in ("fp32", "bf16", "adjoint", "train", "long"):
        K, M, S = case["K"], case["M"], case["S"]
        T = int(_lengths(case, None).sum())
        params = 4 * (K * K + K * M + K)
        if path in ("adjoint", "train"):
            # the forward and backward recursions and the expected transitions: 2 K^2 each a step;
            # the training iteration also writes two further sets of parameters
            return dict(bytes=4 * T + 8 * (S + 1) + 8 * S + params * (2 if path == "adjoint" else 4), flops=6 * K * K * T)
        # parallel in T: the step matrices' products, 2 K^3 a step; else 2 K^2
        return dict(bytes=4 * T + 8 * (S + 1) + 8 * S + params, flops=(2 * K ** 3 if path == "long" else 2 * K * K) * T)
    if path in ("ragged_row", "marshal", "segreduce"):
        S = case["S"]
        N = int(_lengths(case, None).sum())
        size = DTYPES[case.get("dtype", "int32")].itemsize
        if path == "marshal":
            return dict(bytes=2 * size * N + 24 * S, flops=0)
        if path == "ragged_row":     # pieces and tables in, sums, maximum and doubled data out
            return dict(bytes=8 * N + 24 * S, flops=3 * N)
        return dict(bytes=size * N + 16 * S, flops=2 * N)
    if path == "patterns":           # x in; the mapped array, the sum and the loop's array out
        size = DTYPES[case["dtype"]].itemsize
        wide = size if case["dtype"].startswith("float") else 8
        return dict(bytes=case["n"] * (3 * size + wide), flops=6 * case["n"])
    if path == "gravity":
        n = case["n"]
        return dict(bytes=28 * n, flops=20 * n * n)
    n, nb = case["n"], case["nb"]
    pairs = n * nb if nb else n * (n - 1) // 2
    return dict(bytes=12 * (n + nb), flops=5 * pairs)


# --------------------------------------------------------------------------------- exact
def _hmm_exact(s, grads):
    """Scaled forward-backward in 64 bits over the sequences side by side, longest first."""
    A, B, pi = (s[k].detach().double().exp() for k in ("log_A", "log_B", "log_pi"))
    Bt = B.t().contiguous()
    off = s["offsets"].cpu().numpy()
    T = np.diff(off)
    order = np.argsort(-T, kind="stable")
    Ts = T[order]
    Tmax = int(Ts[0])
    n_at = np.searchsorted(-Ts, -np.arange(Tmax), side="left").tolist()      # sequences with T > t
    first = torch.from_numpy(off[:-1][order]).to(DEV)
    S, K = len(T), A.shape[0]
    ll = torch.zeros(S, dtype=torch.float64, device=DEV)
    alphas, scales, syms = [], [], []
    a = None
    for t in range(Tmax):
        n = n_at[t]
        o = s["obs"][first[:n] + t].long()
        a = (pi.expand(n, K) if t == 0 else a[:n] @ A) * Bt[o]
        c = a.sum(1, keepdim=True)
        a = a / c
        ll[:n] += c[:, 0].log()
        if grads:
            alphas.append(a)
            scales.append(c)
            syms.append(o)
    out = torch.empty_like(ll)
    out[torch.from_numpy(order).to(DEV)] = ll
    if not grads:
        return out
    U = torch.zeros_like(A)
    counts = torch.zeros_like(Bt)
    beta = torch.ones(S, K, dtype=torch.float64, device=DEV)
    for t in range(Tmax - 1, -1, -1):
        n = n_at[t]
        if t + 1 < Tmax and n_at[t + 1]:
            m = n_at[t + 1]
            v = Bt[syms[t + 1]] * beta[:m] / scales[t + 1]
            U += alphas[t][:m].t() @ v
            beta[:m] = v @ A.t()
        counts.index_add_(0, syms[t], alphas[t] * beta[:n])
    return out, (A * U, counts.t().contiguous(), (alphas[0] * beta).sum(0))


def _long_exact(s, chunk=500):
    """Products of the step matrices of all chunks side by side, then folded in order."""
    A, B, pi = (s[k].double().exp() for k in ("log_A", "log_B", "log_pi"))
    Bt = B.t().contiguous()
    K = A.shape[0]
    off = s["offsets"].cpu().numpy()
    start, count, where = [], [], []
    for q in range(len(off) - 1):
        where.append(len(start))
        for t in range(int(off[q]) + 1, int(off[q + 1]), chunk):
            start.append(t)
            count.append(min(chunk, int(off[q + 1]) - t))
    first, n = torch.tensor(start, device=DEV), torch.tensor(count, device=DEV)
    X = torch.eye(K, dtype=torch.float64, device=DEV).expand(len(start), K, K).contiguous()
    logs = torch.zeros(len(start), dtype=torch.float64, device=DEV)
    for k in range(chunk):
        on = k < n
        Y = (X @ A) * Bt[s["obs"][torch.where(on, first + k, first)].long()][:, None, :]
        top = Y.amax((1, 2))
        X = torch.where(on[:, None, None], Y / top[:, None, None], X)
        logs += torch.where(on, top.log(), 0.0)
    out = []
    for q in range(len(off) - 1):
        v = pi * Bt[int(s["obs"][int(off[q])])]
        total = torch.zeros((), dtype=torch.float64, device=DEV)
        for c in range(where[q], where[q + 1] if q + 1 < len(where) else len(start)):
            v = v @ X[c]
            total = total + v.sum().log() + logs[c]
            v = v / v.sum()
        out.append(total + v.sum().log())
    return torch.stack(out)


def exact(case, seed):
    path = case["path"]
    s = prepare(case, seed)
    if path in ("fp32", "bf16"):
        return _hmm_exact(s, False)
    if path == "long":
        return _long_exact(s)
    if path == "adjoint":
        ll, g = _hmm_exact(s, True)
        return (*g, ll)
    if path == "train":
        ll, g = _hmm_exact(s, True)
        p = [s[k].detach().double() for k in ("log_A", "log_B", "log_pi")]
        total = [t.sum(-1, keepdim=True) for t in g]
        return dict(ll=ll, grad=g, theta=tuple(t - q.softmax(-1) * u for t, q, u in zip(g, p, total)),
                    new=tuple((t / u).log() for t, u in zip(g, total)))
    if path in ("ragged_row", "marshal"):
        t = s["table"]
        flat = torch.cat(t.seqs)
        off = torch.from_numpy(_offsets(_lengths(case, seed))).to(DEV)
        if path == "marshal":
            return flat, off
        sums = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), (flat.long() ** 2 + 1).cumsum(0)])
        seg = sums[off[1:]] - sums[off[:-1]]
        return seg, seg.max().reshape(1), 2 * flat
    if path == "segreduce":
        x = s["data"]
        x = x.double() if x.dtype.is_floating_point else x.long()
        kind = case["map"]
        x = x * x + 1 if kind == "sq_plus_one" else x.abs() if kind == "abs" else x * 3 if kind == "scale" else x
        S = case["S"]
        ids = torch.repeat_interleave(torch.arange(S, device=DEV), s["offsets"].diff())
        inf = torch.iinfo(torch.int64).max if x.dtype == torch.int64 else math.inf
        ninf = torch.iinfo(torch.int64).min if x.dtype == torch.int64 else -math.inf
        out = torch.full((S,), {"add": 0, "min": inf, "max": ninf}[case["op"]], dtype=x.dtype, device=DEV)
        return out.scatter_reduce_(0, ids, x, {"add": "sum", "min": "amin", "max": "amax"}[case["op"]])
    if path == "patterns":
        x = s["x"].double() if s["x"].dtype.is_floating_point else s["x"].long()
        y = x * x + 1
        return y, x + x, y.sum().reshape(1), 2 * x
    if path == "gravity":
        p = s["aos"].double()
        out = []
        for i in range(0, case["n"], 512):
            d = [p[None, :, k] - p[i:i + 512, None, k] for k in range(3)]
            w = p[None, :, 3] * (d[0] ** 2 + d[1] ** 2 + d[2] ** 2 + case["eps"] ** 2) ** -1.5
            out.append(torch.stack([(w * q).sum(1) for q in d]))
        return tuple(torch.cat(out, 1))
    # whole numbers: the products and sums rounded to 32 bits one by one, as the call promises
    A, B = s["A"], s["B"] if s["B"] is not None else s["A"]
    rising = s["edges"].flip(0).contiguous().to(DEV)
    n = len(rising)

    def bins(d):
        return torch.bincount((n - torch.searchsorted(rising, d.reshape(-1))), minlength=n + 1)

    hist = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    for i in range(0, len(A), 512):
        x, y, z = (A[i:i + 512, None, k] * B[None, :, k] for k in range(3))
        hist += bins((x + y) + z)
    if s["B"] is None:
        hist = (hist - bins((A[:, 0] * A[:, 0] + A[:, 1] * A[:, 1]) + A[:, 2] * A[:, 2])) // 2
    return hist
