"""The work a user of this library has it do, as a list of cases that a timing
program runs through the public Python entry points.

A user quantises float features (`boruta_quantise`), then either steps a
`Session` one Boruta iteration at a time (checkpointing its state between
iterations), or calls `boruta_fit` / `boruta_fit_batch` for whole runs.  The
cases span the sizes of the repository's own workloads: the paper-size
problem (N = 1000, p = 50), the paper's regression study, the wide binary,
SNP and N = 1e6 multiclass workloads of the benchmark, and uneven batches;
both importances in both of Alg. 3's forms, both precisions and tie rules,
plain and graph-replayed iterations, 2 to 8 classes and regression, odd sizes.

`exact` restates the method in plain torch with 64-bit numbers (integers for
counts, draws and target sums; float64 for scores, losses and statistics).
"""
import math

import numpy as np
import torch

from paper_2605_09950_gb300 import boruta

DEV = "cuda"


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # paper-size features on their way in: one small upload is quantised
        dict(name="quantise_small", kind="quantise", data="gauss", N=1000, p=50, bins=64, classes=2),
        # the benchmark's N = 1e6 matrix on its way in
        dict(name="quantise_large", kind="quantise", data="toeplitz", N=1_000_000, p=500, bins=256, classes=5),
        # one iteration of the paper-size binary problem: launches and latency
        dict(name="step_small", kind="step", data="gauss", N=1000, p=50, bins=64, classes=2, trees=100, depth=8, mtry=0,
             permut=0, form=0, precision=0, tie=0, graph=0, iters=20),
        # a whole small run with everything a call pays for (setup, iterations
        # replayed from a graph, results), odd sizes
        dict(name="fit_small_graph", kind="fit", data="gauss", N=1003, p=47, bins=64, classes=2, trees=100, depth=8,
             mtry=0, permut=1, form=0, precision=1, tie=1, graph=1, iters=20),
        # the paper's synthetic regression study: every column tried at every split
        dict(name="step_paper_regression", kind="step", data="paper", N=10_000, p=50, bins=128, classes=0, trees=100,
             depth=16, mtry=1 << 20, permut=1, form=0, precision=0, tie=1, graph=0, iters=4),
        # Alg. 3 as printed, on a small three-class problem of odd size
        dict(name="step_printed_form", kind="step", data="gauss", N=5003, p=61, bins=128, classes=3, trees=100, depth=10,
             mtry=0, permut=1, form=1, precision=0, tie=1, graph=0, iters=4),
        # eight classes, impurity importance, ragged sizes
        dict(name="step_eight_classes", kind="step", data="gauss", N=30_011, p=203, bins=200, classes=8, trees=100,
             depth=14, mtry=0, permut=0, form=0, precision=0, tie=1, graph=0, iters=4),
        # the wide binary workload of the benchmark
        dict(name="step_binary_wide", kind="step", data="gauss", N=100_000, p=1000, bins=256, classes=2, trees=500,
             depth=16, mtry=0, permut=1, form=0, precision=1, tie=0, graph=0, iters=4),
        # the SNP regression workload at a quarter of its columns
        dict(name="step_snp", kind="step", data="snp", N=20_000, p=5003, bins=256, classes=0, trees=100, depth=12, mtry=0,
             permut=0, form=0, precision=0, tie=0, graph=0, iters=4),
        # many independent problems of uneven size, as one call
        dict(name="fit_batch", kind="batch", data="gauss", N=50_000, p=2500, bins=128, classes=4, trees=200, depth=10,
             mtry=0, permut=1, form=0, precision=1, tie=0, graph=0, iters=3, jobs=12),
        # the benchmark's default workload: the largest
        dict(name="step_multiclass_large", kind="step", data="toeplitz", N=1_000_000, p=500, bins=256, classes=5,
             trees=300, depth=20, mtry=0, permut=1, form=0, precision=1, tie=0, graph=0, iters=4),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind of call, then sizes over its whole range (a
    case's estimated work stays below a third of the largest listed one's)."""
    kind = rng.choice(["quantise", "step", "step", "step", "step", "fit", "batch"])
    if kind == "quantise":
        N = _logu(rng, 300, 1_000_000)
        return dict(kind="quantise", data="gauss", N=N, p=min(_logu(rng, 5, 4000), max(5, 400_000_000 // N)),
                    bins=rng.randint(2, 256), classes=rng.randint(2, 5))
    data = rng.choice(["gauss", "gauss", "gauss", "toeplitz", "snp", "paper"]) if kind == "step" else "gauss"
    c = dict(kind=kind, data=data, N=_logu(rng, 500, 400_000), p=_logu(rng, 20, 2000), bins=rng.choice([32, 64, 128, 256, 256]),
             classes=rng.randint(2, 8), trees=_logu(rng, 30, 300), depth=rng.randint(4, 18), mtry=0, permut=rng.randint(0, 1),
             form=0, precision=rng.randint(0, 1), tie=rng.randint(0, 1), graph=0, iters=4)
    if data == "toeplitz":
        c.update(classes=rng.randint(3, 5), bins=256)
    elif data == "snp":
        c.update(classes=0, bins=256, N=_logu(rng, 1000, 30_000), p=_logu(rng, 200, 6000), depth=rng.randint(6, 12))
    elif data == "paper":
        c.update(classes=0, bins=128, p=50, N=_logu(rng, 2000, 20_000), mtry=rng.choice([0, 1 << 20]))
    if kind == "step" and rng.random() < 0.15:  # Alg. 3 as printed, on small problems
        c.update(permut=1, form=1, N=min(c["N"], 8000), p=min(c["p"], 100))
    if kind == "fit":
        c.update(N=_logu(rng, 500, 5000), p=_logu(rng, 20, 200), depth=rng.randint(4, 10), iters=rng.randint(5, 20),
                 graph=rng.randint(0, 1))
    if kind == "batch":
        c.update(N=_logu(rng, 2000, 50_000), p=_logu(rng, 100, 2500), classes=4, bins=128, trees=_logu(rng, 50, 200),
                 depth=rng.randint(6, 10), iters=2, jobs=rng.randint(4, 12))
    while _adds(c) > 4e10:
        c["trees"] = max(10, c["trees"] * 2 // 3)
        if c["trees"] == 10:
            c["N"] = max(500, c["N"] * 2 // 3)
    return c


def _p_aug(p):
    s = p
    while s < 5:
        s *= 2
    return p + s


def _mtry(c):
    pa = _p_aug(c["p"])
    return min(c["mtry"], pa) if c["mtry"] else max(1, pa // 3 if c["classes"] == 0 else math.isqrt(pa))


def _adds(c):
    """Histogram adds of one iteration: every in-bag row once per sampled
    column and level (at most the depth a tree of N rows can use)."""
    levels = min(c["depth"], max(1, int(math.log2(c["N"]))))
    return c["trees"] * 0.632 * c["N"] * _mtry(c) * levels


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: the
    histogram adds of the fit (quantise: a binary search per value)."""
    N, p = case["N"], case["p"]
    if case["kind"] == "quantise":
        return {"bytes": 5.0 * N * p, "flops": float(N) * p * math.ceil(math.log2(case["bins"]))}
    iters = 1 if case["kind"] == "step" else case["iters"]
    ybytes = 8 if case["classes"] == 0 else 1
    one = float(N) * p + ybytes * N + iters * p * 8 + 5 * p
    if case["kind"] == "batch":
        per = [dict(case, N=n, p=q) for n, q, _ in _batch_shapes(case)]
        return {"bytes": sum(float(c["N"]) * c["p"] + c["N"] + iters * c["p"] * 8 for c in per),
                "flops": iters * sum(_adds(c) for c in per)}
    return {"bytes": one, "flops": iters * _adds(case)}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _features(case, g, N, p, classes):
    """(list of float32 column blocks [q, N], y): class-conditional Gaussians
    with informative and collinear columns, or AR(1) blocks with softmax labels."""
    if case["data"] == "toeplitz":
        logits = torch.zeros(classes, N, device=DEV)
        blocks, n_inf, done = [], min(25, (p + 9) // 10), 0
        W = torch.randn(classes, n_inf, generator=g, device=DEV) / math.sqrt(n_inf)
        for b in range((p + 9) // 10):
            q = min(10, p - done)
            F = torch.randn(q, N, generator=g, device=DEV)
            for j in range(1, q):
                F[j] = 0.8 * F[j - 1] + 0.6 * F[j]
            if b < n_inf:
                logits += W[:, b:b + 1] * F[0]
            blocks.append(F)
            done += q
        u = torch.rand(N, generator=g, device=DEV)
        y = (u[None, :] > torch.softmax(logits, 0).cumsum(0)).sum(0).clamp(max=classes - 1).to(torch.uint8)
        return blocks, y
    y = torch.randint(0, classes, (N,), generator=g, device=DEV, dtype=torch.uint8)
    y[:classes] = torch.arange(classes, device=DEV, dtype=torch.uint8)  # every class is present
    F = torch.randn(p, N, generator=g, device=DEV)
    order = torch.randperm(p, generator=g, device=DEV)
    n_inf = min(p, max(3, p // 25 if p >= 500 else p // 5))
    mu = (torch.rand(n_inf, classes, generator=g, device=DEV) < 0.5).float()
    mu[:, 0] = 0.0
    F[order[:n_inf]] += mu[:, y.long()]
    n_lin = min(max(0, p - n_inf), p // 25)  # collinear columns: weighted sums of informative ones
    for k in range(n_lin):
        src = order[torch.randint(0, n_inf, (4,), generator=g, device=DEV)]
        F[order[n_inf + k]] = (torch.tensor([0.1, 0.2, 0.3, 0.4], device=DEV) @ F[src]
                               + 0.1 * torch.randn(N, generator=g, device=DEV))
    return [F], y


def _paper(g, N, p):
    """The paper's synthetic regression data (its first 50 columns)."""
    F = torch.rand(p, N, generator=g, device=DEV, dtype=torch.float64)
    x = lambda i: F[i - 1]
    y = (5 * x(27) ** 3 + 4 * x(49) ** 2 + 5 * x(31) * x(46) + 2 * x(14) - 2.5 * x(40) + 3.5 * x(18) ** (1.0 / 3.0)
         + torch.exp(x(20)) + 2 * torch.sin(3.14 * x(26)) + 5 * torch.cos(3.14 * x(33)))
    y = y + math.sqrt(1e-5) * torch.randn(N, generator=g, device=DEV, dtype=torch.float64)
    return F.float(), torch.round(y * 2.0**20).to(torch.int64)


def _snp(g, N, p):
    """Genotypes Bin(2, f) and a polygenic trait in units of 2^-20."""
    f = 0.05 + 0.45 * torch.rand(p, 1, generator=g, device=DEV)
    X = torch.zeros(p, (N + 15) // 16 * 16, dtype=torch.uint8, device=DEV)
    for _ in range(2):
        X[:, :N] += (torch.rand(p, N, generator=g, device=DEV) < f).to(torch.uint8)
    n = min(p, 50)
    cols = torch.randperm(p, generator=g, device=DEV)[:n]
    G = X[cols, :N].double()
    beta = torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    y = (beta[:, None] * G).sum(0) + torch.randn(N, generator=g, device=DEV, dtype=torch.float64)
    for k in range(0, n - 1, 5):
        y = y + beta[k] * G[k] * G[k + 1]
    return X, torch.round(y * 2.0**20).to(torch.int64)


def _inputs(case, seed, quantise, N=None, p=None, classes=None):
    """(X bins [p, ld], y) of a problem; quantise(F, n_bins) bins float columns."""
    g = _gen(seed)
    N, p = N or case["N"], p or case["p"]
    if case["data"] == "snp":
        return _snp(g, N, p)
    if case["data"] == "paper":
        F, y = _paper(g, N, p)
        return quantise(F, case["bins"]), y
    blocks, y = _features(case, g, N, p, classes or case["classes"])
    X = torch.zeros(p, (N + 15) // 16 * 16, dtype=torch.uint8, device=DEV)
    at = 0
    while blocks:
        take = blocks[:64]
        blocks = blocks[64:]
        F = torch.cat(take) if len(take) > 1 else take[0]
        X[at:at + F.shape[0]] = quantise(F, case["bins"])
        at += F.shape[0]
    return X, y


def _batch_shapes(case):
    """(N, p, classes) of each job: uneven, spread evenly over the logarithm
    from a hundredth of the case's N and p up to them, in different orders."""
    n, out = case["jobs"], []
    for j in range(n):
        u, v = j / max(1, n - 1), ((j * 5 + 3) % n) / max(1, n - 1)
        out.append((max(200, int(case["N"] * 0.01 ** (1 - u))), max(10, int(case["p"] * 0.01 ** (1 - v))),
                    2 + j % (case["classes"] - 1)))
    return out


def _task(case):
    return (boruta.REGRESSION if case["classes"] == 0 else boruta.CLASSIFICATION) | (boruta.PERMUT if case["permut"] else 0)


def _options(case):
    return dict(precision=case["precision"], tie_break=case["tie"], graph=case["graph"], permut_form=case["form"])


def prepare(case, seed):
    if case["kind"] == "quantise":
        blocks, _ = _features(case, _gen(seed), case["N"], case["p"], case["classes"])
        F = torch.cat(blocks) if len(blocks) > 1 else blocks[0]
        return dict(kind="quantise", F=F, bins=case["bins"])
    args = dict(task=_task(case), n_trees=case["trees"], max_depth=case["depth"], mtry=case["mtry"], n_bins=case["bins"],
                max_iter=case["iters"], alpha=0.01, seed=int(seed))
    quantise = boruta.boruta_quantise
    if case["kind"] == "batch":
        jobs = []
        for j, (N, p, C) in enumerate(_batch_shapes(case)):
            X, y = _inputs(case, seed * 100 + j, quantise, N, p, C)
            jobs.append(dict(args, X=X, y=y, N=N, n_classes=C, seed=int(seed) * 1000 + j))
        return dict(kind="batch", jobs=jobs, options=_options(case))
    X, y = _inputs(case, seed, quantise)
    if case["kind"] == "fit":
        return dict(kind="fit", args=dict(args, X=X, y=y, N=case["N"]), options=_options(case))
    S = boruta.Session(X, y, N=case["N"], **args, **_options(case))
    return dict(kind="step", session=S, start=S.read())


def run(state):
    if state["kind"] == "quantise":
        return boruta.boruta_quantise(state["F"], state["bins"])
    if state["kind"] == "fit":
        return boruta.boruta_fit(**state["args"], **state["options"])
    if state["kind"] == "batch":
        return boruta.boruta_fit_batch(state["jobs"], **state["options"])
    S = state["session"]
    S.write(state["start"])  # resume from the checkpoint, run one iteration, checkpoint
    S.step()
    return S.read()


# ---------------------------------------------------------------- the same in plain torch, 64 bits

M32 = 0xFFFFFFFF


def exact(case, seed):
    if case["kind"] == "quantise":
        blocks, _ = _features(case, _gen(seed), case["N"], case["p"], case["classes"])
        F = torch.cat(blocks) if len(blocks) > 1 else blocks[0]
        return _ranks(F, case["bins"])
    if case["kind"] == "batch":
        return None
    iters = 1 if case["kind"] == "step" else case["iters"]
    K, snp = max(1, case["classes"]), case["data"] == "snp"  # three bins: the additions below meet on few cells
    cells = case["trees"] * 2.0 ** min(case["depth"], math.log2(case["N"])) * _mtry(case) * (3 if snp else case["bins"])
    walks = case["trees"] * case["N"] * _p_aug(case["p"]) * case["depth"] if case["permut"] else 0
    if iters * (_adds(case) * (1 + K) * (20 if snp else 1) + cells * K + 3 * walks) > 6e10:
        return None
    X, y = _inputs(case, seed, _ranks)
    return _boruta(case, X[:, :case["N"]].long(), y.long(), int(seed), iters)


def _ranks(F, bins):
    """bin = min(B - 1, floor(B * (number of smaller values) / N))"""
    p, N = F.shape
    out = torch.zeros(p, (N + 15) // 16 * 16, dtype=torch.uint8, device=DEV)
    for j in range(0, p, max(1, (1 << 25) // N)):
        f = F[j:j + max(1, (1 << 25) // N)].contiguous()
        rank = torch.searchsorted(torch.sort(f, 1).values, f, right=False)
        out[j:j + f.shape[0], :N] = (bins * rank // N).clamp(max=bins - 1).to(torch.uint8)
    return out


def _mul32(a, m):
    """(high, low) 32 bits of a * m for a, m in [0, 2^32) held as int64"""
    lo, hi = (a & 0xFFFF) * m, (a >> 16) * m
    mid = (lo >> 16) + (hi & 0xFFFF)
    return (hi >> 16) + (mid >> 16), ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)


def _philox(c0, c1, c2, c3, seed):
    k0, k1 = seed & M32, (seed >> 32) & M32
    c0, c1, c2, c3 = torch.broadcast_tensors(*(torch.as_tensor(c, dtype=torch.int64, device=DEV) for c in (c0, c1, c2, c3)))
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        ah, al = _mul32(c0, 0xD2511F53)
        bh, bl = _mul32(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = bh ^ c1 ^ k0, bl, ah ^ c3 ^ k1, al
    return c0, c1, c2, c3


def _fmix(h):
    h = _mul32(h ^ (h >> 16), 0x85EBCA6B)[1]
    h = _mul32(h ^ (h >> 13), 0xC2B2AE35)[1]
    return h ^ (h >> 16)


def _perm(n, seed, w1, w2, w3, count):
    """The first `count` images of keyed permutations of [0, n): one row per
    entry of w1 / w2 (8-round Feistel network, cycle walking)."""
    half = 1
    while 4**half < n:
        half += 1
    mask = (1 << half) - 1
    keys = _philox(0, w1, w2, w3, seed) + _philox(1, w1, w2, w3, seed)

    def once(x, K):
        left, right = x >> half, x & mask
        for k in K:
            left, right = right, left ^ (_fmix(right ^ k) & mask)
        return (left << half) | right

    x = torch.arange(count, device=DEV).expand(keys[0].numel(), count)
    if n <= 1:
        return x.clone()
    x = once(x, [k.reshape(-1, 1) for k in keys])
    while True:
        row, col = torch.nonzero(x >= n, as_tuple=True)
        if row.numel() == 0:
            return x
        x[row, col] = once(x[row, col], [k.reshape(-1)[row] for k in keys])


def _grow(case, X, y, seed, t, pa):
    """The iteration's trees, level by level: lists over levels of the nodes'
    (split feature or -1, bin, first child, statistics, weight, delta, tree)."""
    N, M, B, tie = X.shape[1], case["trees"], int(X.max()) + 1, case["tie"]
    K = case["classes"] or 1
    unit = (t << 24) + torch.arange(M, device=DEV)
    counts = torch.zeros(M, N, dtype=torch.int64, device=DEV)
    for a in range(0, N, 1 << 16):
        d = torch.arange(a, min(N, a + (1 << 16)), device=DEV)
        lo, hi, _, _ = _philox(d[None, :], 0, unit[:, None], 2 << 24, seed)
        row = (hi * N + (lo * N >> 32)) >> 32  # floor(draw * N / 2^64)
        counts.scatter_add_(1, row, torch.ones_like(row))
    tree, row = torch.nonzero(counts, as_tuple=True)
    w = counts[tree, row]
    value = torch.zeros(row.numel(), K, dtype=torch.int64, device=DEV)
    if case["classes"]:
        value[torch.arange(row.numel(), device=DEV), y[row]] = w
    else:
        value[:, 0] = w * y[row]
    mtry = max(1, min(case["mtry"], pa) if case["mtry"] else (pa // 3 if K == 1 and not case["classes"] else math.isqrt(pa)))
    node, n_nodes = tree.clone(), M
    heap, owner = torch.zeros(M, dtype=torch.int64, device=DEV), torch.arange(M, device=DEV)
    levels = []
    for depth in range(case["depth"] + 1):
        stat = torch.zeros(n_nodes, K, dtype=torch.int64, device=DEV).index_add_(0, node, value)
        n = torch.zeros(n_nodes, dtype=torch.int64, device=DEV).index_add_(0, node, w)
        rows = torch.bincount(node, minlength=n_nodes)
        grow = (rows >= 2) & (depth < case["depth"])
        if case["classes"]:
            grow &= (stat != n[:, None]).all(1)
        feat = torch.full((n_nodes,), -1, dtype=torch.int64, device=DEV)
        bins, delta = torch.zeros_like(feat), torch.zeros(n_nodes, dtype=torch.float64, device=DEV)
        order = torch.argsort(node, stable=True)
        start = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), rows.cumsum(0)])
        active = torch.nonzero(grow).flatten()
        at = 0
        step = max(1, (1 << 27) // (mtry * B * K))
        a_rows = rows[active]
        while at < active.numel():
            end = min(active.numel(), at + step)
            csum = a_rows[at:end].cumsum(0)
            end = at + max(1, int((csum * mtry <= (1 << 27)).sum()))
            ks = active[at:end]
            at = end
            f = _perm(pa, seed, heap[ks], (t << 24) + owner[ks], 3 << 24, mtry)
            if tie == 0:
                f = f.sort(1).values
            m = ks.numel()
            len_k = rows[ks]
            local = torch.repeat_interleave(torch.arange(m, device=DEV), len_k)
            first = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), len_k.cumsum(0)[:-1]])
            e = order[start[ks][local] + torch.arange(local.numel(), device=DEV) - first[local]]
            cell = (local[:, None] * mtry + torch.arange(mtry, device=DEV)) * B + X[f[local], row[e][:, None]]
            nl = torch.zeros(m * mtry * B, dtype=torch.int64, device=DEV)
            nl.index_add_(0, cell.flatten(), w[e][:, None].expand(-1, mtry).flatten())
            nl = nl.view(m, mtry, B).cumsum(2)
            num = torch.zeros(m, mtry, B, dtype=torch.float64, device=DEV)
            for k in range(K):
                sl = torch.zeros(m * mtry * B, dtype=torch.int64, device=DEV)
                sl.index_add_(0, cell.flatten(), value[e, k][:, None].expand(-1, mtry).flatten())
                sl = sl.view(m, mtry, B).cumsum(2)
                num += (sl * n[ks][:, None, None] - stat[ks, k][:, None, None] * nl).double() ** 2
                del sl
            nr = n[ks][:, None, None] - nl
            d = torch.where((nl > 0) & (nr > 0), num / (nl * nr).clamp(min=1).double(), -1.0).view(m, -1)
            best = d.max(1).values
            arg = (d == best[:, None]).double().argmax(1)  # the first of equal scores
            ok = best > 0
            feat[ks] = torch.where(ok, f[torch.arange(m, device=DEV), arg // B], -1)
            bins[ks] = arg % B
            delta[ks] = torch.where(ok, best / n[ks].double(), 0.0)
        split = torch.nonzero(feat >= 0).flatten()
        child = torch.zeros(n_nodes, dtype=torch.int64, device=DEV)
        child[split] = 2 * torch.arange(split.numel(), device=DEV)
        levels.append(dict(feat=feat, bin=bins, child=child, stat=stat, n=n, delta=delta, tree=owner))
        if split.numel() == 0:
            break
        keep = feat[node] >= 0
        node, row, w, value = node[keep], row[keep], w[keep], value[keep]
        right = X[feat[node], row] > bins[node]
        node = child[node] + right
        heap = torch.stack([2 * heap[split] + 1, 2 * heap[split] + 2], 1).flatten()
        owner = owner[split].repeat_interleave(2)
        n_nodes = 2 * split.numel()
    base = 0
    for lv in levels:  # children as indices into all nodes together
        base += lv["feat"].numel()
        lv["child"] = lv["child"] + base
    tr = {k: torch.cat([lv[k] for lv in levels]) for k in levels[0]}
    tr["depth"] = len(levels)
    return tr, counts


def _leaf(tr, X, tree, row, f=-1, flush=None):
    """Leaf of each (tree, row), column f read at the row's flush_index."""
    k = tree.clone()
    for _ in range(tr["depth"]):
        g = tr["feat"][k]
        x = X[g.clamp(min=0), row if flush is None else torch.where(g == f, flush, row)]
        k = torch.where(g < 0, k, tr["child"][k] + (x > tr["bin"][k]))
    return k


def _loss(case, a, b):
    """KL between smoothed class probabilities, or the squared difference of
    means in units of 2^-20."""
    if case["classes"] == 0:
        return ((a - b)[:, 0] * 2.0**-20) ** 2
    eps = 1e-7
    a, b = (a + eps) / (1 + case["classes"] * eps), (b + eps) / (1 + case["classes"] * eps)
    return (a * torch.log(a / b)).sum(1)


def _importance(case, tr, counts, X, seed, t):
    M, N, pa = case["trees"], X.shape[1], X.shape[0]
    if not case["permut"]:
        s = torch.nonzero(tr["feat"] >= 0).flatten()
        imp = torch.zeros(M, pa, dtype=torch.float64, device=DEV)
        imp.index_put_((tr["tree"][s], tr["feat"][s]), tr["delta"][s], accumulate=True)
        total = imp.sum(1, keepdim=True)
        return torch.where(total > 0, imp / total, 0.0)
    pi = _perm(N, seed, torch.zeros(1, dtype=torch.int64, device=DEV), t << 24, 4 << 24, N)[0]
    value = tr["stat"].double() / tr["n"][:, None].double()
    used = torch.unique(tr["feat"])
    if case["form"] == 1:
        tree = torch.arange(M, device=DEV).repeat_interleave(N)
        row = torch.arange(N, device=DEV).repeat(M)
        imp = torch.zeros(1, pa, dtype=torch.float64, device=DEV)
        base = value[_leaf(tr, X, tree, row)].view(M, N, -1).mean(0)
        for f in used[used >= 0].tolist():
            imp[0, f] = _loss(case, base, value[_leaf(tr, X, tree, row, f, pi[row])].view(M, N, -1).mean(0)).mean()
        return imp
    tree, row = torch.nonzero(counts == 0, as_tuple=True)
    oob = torch.bincount(tree, minlength=M).double()
    imp = torch.zeros(M, pa, dtype=torch.float64, device=DEV)
    q = _leaf(tr, X, tree, row)
    for f in used[used >= 0].tolist():
        q2 = _leaf(tr, X, tree, row, f, pi[row])
        loss = torch.where(q == q2, 0.0, _loss(case, value[q], value[q2]))
        imp[:, f] = torch.zeros(M, dtype=torch.float64, device=DEV).index_add_(0, tree, loss) / oob.clamp(min=1)
    return imp


def _boruta(case, X, y, seed, iters):
    p, N = X.shape
    state, hits = np.zeros(p, np.int8), np.zeros(p, np.int32)
    history, smax, t = np.full((case["iters"], p), np.nan), np.full(case["iters"], np.nan), 0
    while t < iters and (state == 0).any():
        t += 1
        live = np.flatnonzero(state >= 0)
        n_sha = len(live)
        while n_sha < 5:
            n_sha *= 2
        cols = torch.as_tensor(live, device=DEV)
        src = cols[torch.arange(n_sha, device=DEV) % len(live)]
        zero = torch.zeros(1, dtype=torch.int64, device=DEV)
        Xa = torch.cat([X[cols]] + [X[src[c], _perm(N, seed, zero, (t << 24) + c, 1 << 24, N)[0]][None] for c in range(n_sha)])
        tr, counts = _grow(case, Xa, y, seed, t, Xa.shape[0])
        imp = _importance(case, tr, counts, Xa, seed, t)
        M = imp.shape[0]
        mean = imp.mean(0)
        if M > 1:
            sd = imp.std(0)
            s = torch.where(sd == 0, torch.where(mean == 0, 0.0, math.inf), mean / (sd / math.sqrt(M)))
        else:
            s = mean
        s = s.cpu().numpy()
        smax[t - 1] = s[len(live):].max()
        history[t - 1, live] = s[:len(live)]
        hits[live] += s[:len(live)] > smax[t - 1]
        m = int((state == 0).sum())
        for j in np.flatnonzero(state == 0):
            above = sum(math.comb(t, k) for k in range(int(hits[j]), t + 1)) / 2**t
            below = sum(math.comb(t, k) for k in range(0, int(hits[j]) + 1)) / 2**t
            state[j] = 1 if above < 0.01 / m else (-1 if below < 0.01 / m else 0)
    return dict(decision=state, hits=hits, imp_history=history, shadow_max=smax, iterations=t)
