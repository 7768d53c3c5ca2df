"""Workloads of the GenCD library, as its users run them.

Each case is one call pattern at one size: a warm-started run of a variant's
iterations on a problem that is resident on the GPU, a regularisation path in
a batch of slots, a cold start from new data, a served stream of requests, or
the allocation-free propose.  Sizes are those of the repository's workloads
(uniform 2,000 x 5,000; the shapes of the paper's two data sets; the Zipf(1.1)
problems of 4e7 and 2e8 non-zeros) and of their ranges.
"""

import math
import types

import numpy as np
import torch

from paper_1206_6409_gb300 import binding as gb

DEV = "cuda"


def listed():
    return [
        # the 2,000 x 5,000 problem with the paper's asynchronous variant (P is
        # its P*): one iteration is a few microseconds of work, so launches
        # and latency are what a user waits for
        dict(name="shotgun-small-f64", kind="run", variant="shotgun", precision="f64", loss="logistic", law="uniform",
             values="pm1", n=2000, k=5000, per_col=20, P=375, blocks=0, iters=50, lam=0.01),
        # the same data with one distance-2 colour class per iteration
        dict(name="coloring-small-f64", kind="run", variant="coloring", precision="f64", loss="squared", law="uniform",
             values="pm1", n=2000, k=5000, per_col=20, P=0, blocks=0, iters=200, lam=0.01),
        # the shape of DOROTHEA (binary drug-discovery data): few rows, many
        # short columns, the single best column per iteration
        dict(name="greedy-binary-dorothea", kind="run", variant="greedy", precision="binary", loss="logistic",
             law="uniform", values="binary", n=800, k=100000, per_col=7, P=0, blocks=0, iters=20, lam=0.05),
        # the shape of REUTERS (tf-idf text): rows that fit one slab of u,
        # values stored in bfloat16
        dict(name="tg-bf16-reuters", kind="run", variant="thread_greedy", precision="bf16", loss="logistic",
             law="uniform", values="lognormal", n=23865, k=47237, per_col=37, P=0, blocks=512, iters=20, lam=0.05),
        # text-like columns in double precision
        dict(name="tg-f64-zipf-20M", kind="run", variant="thread_greedy", precision="f64", loss="logistic", law="zipf",
             values="lognormal", n=100003, k=399989, nnz=20_000_000, cap=5000, P=0, blocks=128, iters=10, lam=0.05),
        # the Lasso of the regularisation-path workload, one warm start; few
        # partitions, as its solves back off to
        dict(name="tg-f32-zipf-40M", kind="run", variant="thread_greedy", precision="f32", loss="squared", law="zipf",
             values="lognormal", n=200000, k=500000, nnz=40_000_000, cap=10000, P=0, blocks=16, iters=10, lam=0.05),
        # the throughput workload at its full size
        dict(name="tg-f32-zipf-200M", kind="run", variant="thread_greedy", precision="f32", loss="logistic",
             law="zipf", values="lognormal", n=1000000, k=4000000, nnz=200_000_000, cap=50000, P=0, blocks=1024,
             iters=10, lam=0.05),
        # Shotgun at the parallelism the paper quotes for REUTERS, on text-like
        # columns of 1 to 5,000 non-zeros
        dict(name="shotgun-f32-zipf-20M", kind="run", variant="shotgun", precision="f32", loss="logistic", law="zipf",
             values="lognormal", n=100000, k=400000, nnz=20_000_000, cap=5000, P=800, blocks=0, iters=20, lam=0.05),
        # cross-validation: chains over folds and lambda grids, one slot each
        dict(name="path-32-slots", kind="path", loss="logistic", law="zipf", values="lognormal", n=20000, k=50000,
             nnz=4_000_000, cap=1000, folds=5, slots=32, chains=32, nlambda=2, blocks=128, iters=30, lam=0.1),
        # the propose of a caller that cannot allocate
        dict(name="noalloc-f64", kind="noalloc", loss="logistic", law="zipf", values="lognormal", n=60000, k=150000,
             nnz=6_000_000, cap=3000, lam=0.05),
        # a cold start: new data on the device, one iteration, w back
        dict(name="create-f32-zipf-20M", kind="create", variant="thread_greedy", precision="f32", loss="logistic",
             law="zipf", values="lognormal", n=100000, k=400000, nnz=20_000_000, cap=5000, P=0, blocks=1024, iters=1,
             lam=0.05),
        # a burst of independent requests from host memory, served in slots
        dict(name="serve-8", kind="serve", nreq=8, slots=4, loss="logistic", n=3000, k=9001, per_col=31, blocks=64,
             iters=100, lam=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))


def _parallel(n, k, nnz):
    """About P*, the number of columns that may move at once (k over twice the
    Gram matrix's largest eigenvalue): for positive unit-norm columns that is
    the rank-one part, about 0.36 of the rows' mean degree, plus the noise."""
    return max(1, int(k / (2.0 * (0.36 * nnz / n + (1.0 + math.sqrt(k / n)) ** 2))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "run", "path", "noalloc", "create", "serve"])
    loss = rng.choice(["squared", "logistic"])
    # the squared loss has no slack in its curvature bound: best columns moved
    # together overshoot and, over many steps, diverge unless they are few
    few = rng.choice([1, 2, 3]) if loss == "squared" else 0
    if kind == "serve":
        return dict(kind="serve", nreq=rng.randint(2, 8), slots=rng.choice([1, 2, 4, 8]), loss=loss,
                    n=_log(rng, 1000, 6000), k=_log(rng, 1000, 20000), per_col=rng.randint(5, 60),
                    blocks=few or rng.choice([16, 64]), iters=10 * rng.randint(5, 10), lam=rng.choice([0.1, 0.2]))
    if kind == "path":
        n, k = _log(rng, 2000, 30000), _log(rng, 3000, 60000)
        slots = rng.choice([5, 8, 16, 20, 32, 64])
        return dict(kind="path", loss=loss, law="zipf", values="lognormal", n=n, k=k,
                    nnz=_log(rng, 10 * k, min(80 * k, 4_000_000)), cap=max(50, n // 20), folds=rng.choice([3, 5]),
                    slots=slots, chains=slots, nlambda=rng.choice([1, 2, 3]), blocks=few or rng.choice([32, 128]),
                    iters=10 * rng.randint(1, 4), lam=0.1)
    if kind == "noalloc":
        n, k = _log(rng, 1000, 300000), _log(rng, 1000, 500000)
        return dict(kind="noalloc", loss=loss, law="zipf", values="lognormal", n=n, k=k,
                    nnz=_log(rng, 5 * k, min(60 * k, 30_000_000)), cap=max(50, n // 20), lam=0.05)
    if kind == "create":
        n, k = _log(rng, 1000, 300000), _log(rng, 2000, 1_000_000)
        return dict(kind="create", variant="thread_greedy", precision=rng.choice(["f64", "f32", "bf16"]), loss=loss,
                    law="zipf", values="lognormal", n=n, k=k, nnz=_log(rng, 10 * k, min(80 * k, 40_000_000)),
                    cap=max(50, n // 20), P=0, blocks=1024, iters=1, lam=0.05)
    variant = rng.choice(["thread_greedy", "thread_greedy", "thread_greedy", "greedy", "shotgun", "coloring"])
    precision = rng.choice(["f64", "f32", "bf16", "binary"])
    case = dict(kind="run", variant=variant, precision=precision, loss=loss, P=0, blocks=0,
                values="binary" if precision == "binary" else "lognormal", lam=rng.choice([0.02, 0.05, 0.1]))
    if variant == "coloring":  # a colouring visits the neighbours of every entry: moderate row degrees
        k = _log(rng, 1000, 20000)
        return dict(case, law="uniform", n=max(k // 4, _log(rng, 1000, 20000)), k=k, per_col=rng.randint(3, 24),
                    iters=10 * rng.randint(5, 30))
    if variant == "shotgun":
        n, k, per_col = _log(rng, 2000, 200000), _log(rng, 4000, 500000), rng.randint(5, 60)
        return dict(case, law=rng.choice(["uniform", "zipf"]), n=n, k=k, per_col=per_col, cap=max(50, n // 20),
                    P=_log(rng, 2, min(1000, _parallel(n, k, per_col * k))), iters=10 * rng.randint(2, 8))
    n, k = _log(rng, 800, 1_000_000), _log(rng, 2000, 3_000_000)
    if rng.random() < 0.4:
        per_col = rng.randint(2, min(60, max(3, 90_000_000 // k)))
        case.update(law="uniform", n=n, k=k, per_col=per_col)
        nnz = per_col * k
    else:
        nnz = _log(rng, 8 * k, min(80 * k, 90_000_000))
        case.update(law="zipf", n=n, k=k, nnz=nnz, cap=max(50, n // 20))
    # the best columns of the partitions are more alike than random ones: fewer than P*
    most = 1 + _parallel(n, k, nnz) // (64 if loss == "squared" else 8)
    return dict(case, blocks=min(rng.choice([16, 64, 200, 1024]), most), iters=10)


# ---------------------------------------------------------------------------
# inputs: a sparse column-major X with a planted model, from the seed alone

def _zipf_counts(k, nnz, cap):
    """Column lengths clamp(round(C r^-1.1), 1, cap) by rank, C by bisection."""
    r = torch.arange(1, k + 1, dtype=torch.float64, device=DEV).pow_(-1.1)
    lo, hi = 0.0, float(nnz) * 10.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        if (r * mid).round_().clamp_(1, cap).sum().item() < nnz:
            lo = mid
        else:
            hi = mid
    return (r * hi).round_().clamp_(1, cap).to(torch.int64)


def _segment_sums(v, counts):
    return torch.segment_reduce(v, "sum", lengths=counts, unsafe=True, axis=0, initial=0.0)


def _entries_of(col_ptr, cols):
    """(positions of the columns' entries, entry counts) in column order."""
    s, cnt = col_ptr[cols], col_ptr[cols + 1] - col_ptr[cols]
    first = torch.cumsum(cnt, 0) - cnt
    pos = torch.arange(int(cnt.sum()), device=cols.device) + torch.repeat_interleave(s - first, cnt)
    return pos, cnt


def _data(case, seed):
    """X (rows sorted and distinct in a column), y, a planted w* and lambda.

    Values: +-1; one value 1/sqrt(nnz_j) per column (binary, unit norm); or
    log-normal with unit-norm columns.  y = sign(X w* + noise) or X w* + noise
    (noise a tenth of the signal).  lambda is a fraction of the smallest one
    that keeps w = 0."""
    n, k = case["n"], case["k"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1_000_003 * int(seed) + n + 7 * k)
    if case["law"] == "zipf":
        nnz = case["nnz"] if "nnz" in case else case["per_col"] * k
        counts = _zipf_counts(k, nnz, min(case["cap"], n))[torch.randperm(k, generator=gen, device=DEV)]
    else:
        counts = torch.full((k,), min(case["per_col"], n), dtype=torch.int64, device=DEV)
    col = torch.repeat_interleave(torch.arange(k, device=DEV), counts)
    key = col.mul_(n).add_(torch.randint(n, (col.numel(),), generator=gen, device=DEV))
    key = torch.unique_consecutive(key.sort().values)  # distinct rows: a column may lose a few entries
    col = key // n
    row = (key - col * n).to(torch.int32)
    counts = torch.bincount(col, minlength=k)
    del key, col
    col_ptr = torch.zeros(k + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=col_ptr[1:])
    nnz = row.numel()
    if case["values"] == "pm1":
        val = torch.randint(0, 2, (nnz,), generator=gen, device=DEV).mul_(2).sub_(1).to(torch.float64)
    elif case["values"] == "binary":
        val = torch.repeat_interleave(counts.double().rsqrt(), counts)
    else:
        val = torch.randn(nnz, generator=gen, device=DEV, dtype=torch.float64).exp_()
        val *= torch.repeat_interleave(_segment_sums(val * val, counts).rsqrt(), counts)
    # planted model: its entries are few, so X w* is summed on the host, in order
    planted = torch.randperm(k, generator=gen, device=DEV)[: max(20, min(2000, k // 100))].sort().values
    wp = torch.randn(planted.numel(), generator=gen, device=DEV, dtype=torch.float64)
    pos, cnt = _entries_of(col_ptr, planted)
    t = np.bincount(row[pos].cpu().numpy(), weights=(val[pos] * torch.repeat_interleave(wp, cnt)).cpu().numpy(),
                    minlength=n)
    t = torch.from_numpy(t).to(DEV)
    y = t + 0.1 * float(np.sqrt(float((t * t).mean()))) * torch.randn(n, generator=gen, device=DEV,
                                                                       dtype=torch.float64)
    if case["loss"] == "logistic":
        y = torch.where(y >= 0, 1.0, -1.0).to(torch.float64)
    w0 = torch.zeros(k, dtype=torch.float64, device=DEV)
    w0[planted] = 0.5 * wp  # a warm start, as from the previous lambda of a path
    u0 = -0.5 * y if case["loss"] == "logistic" else -y
    g0 = _segment_sums(val * u0[row], counts).abs().max().item() / n
    if case.get("precision", "f32" if case["kind"] in ("path", "serve") else "f64") != "f64":
        val = val.to(torch.float32)
    return types.SimpleNamespace(n=n, k=k, nnz=nnz, col_ptr=col_ptr, row_idx=row, val=val, y=y, w0=w0,
                                 loss=case["loss"], lam=case["lam"] * g0)


def _problem(case, d):
    p = gb.Problem(n=d.n, k=d.k, col_ptr=d.col_ptr, row_idx=d.row_idx, val=d.val, y=d.y, loss=d.loss,
                   precision=case["precision"])
    p.set_lambda(d.lam)
    p.set_params(variant=case["variant"], blocks=case["blocks"], P=case["P"])
    return p


def _path_grid(case, d):
    """Chains go over the folds in turn, each with its own run of lambdas."""
    c, q = np.arange(case["chains"])[:, None], np.arange(case["nlambda"])[None, :]
    held_out = (np.arange(case["chains"]) % case["folds"]).astype(np.int32)
    return held_out, d.lam * 0.97 ** c * 0.8 ** q


def _fold(case):
    return (torch.arange(case["n"], device=DEV) % case["folds"]).to(torch.uint8)


def _requests(case, seed):
    out = []
    for q in range(case["nreq"]):
        c = dict(case, law="uniform", values="lognormal", n=case["n"] + 97 * q, k=case["k"] + 211 * q)
        d = _data(c, 64 * int(seed) + q)
        out.append(types.SimpleNamespace(n=d.n, k=d.k, nnz=d.nnz, loss=d.loss, col_ptr=d.col_ptr.cpu().numpy(),
                                         row_idx=d.row_idx.cpu().numpy(), val=d.val.cpu().numpy(),
                                         y=d.y.cpu().numpy()))
    return out


def prepare(case, seed):
    s = types.SimpleNamespace(case=case, kind=case["kind"])
    if s.kind == "serve":
        s.problems = _requests(case, seed)
        s.fracs, s.arrivals = [case["lam"]] * case["nreq"], [0.0] * case["nreq"]
        return s
    d = s.d = _data(case, seed)
    if s.kind == "run":
        s.p = _problem(case, d)
        s.w = torch.empty_like(d.w0)
        if case["variant"] == "coloring":
            s.p.color()
        s.p.set_w(d.w0)
    elif s.kind == "path":
        s.stream = torch.cuda.Stream()
        torch.cuda.synchronize()  # the inputs were made on another stream
        s.b = gb.Batch(d, fold=_fold(case), nfolds=case["folds"], slots=case["slots"], stream=s.stream.cuda_stream)
        s.b.set_params(variant="thread_greedy", blocks=case["blocks"], max_iter=case["iters"], tol_kkt=0.0)
        s.held_out, s.lams = _path_grid(case, d)
    elif s.kind == "noalloc":
        s.z = torch.zeros(d.n, dtype=torch.float64, device=DEV)
        cols = torch.nonzero(d.w0).flatten()
        pos, cnt = _entries_of(d.col_ptr, cols)
        s.z += torch.from_numpy(np.bincount(
            d.row_idx[pos].cpu().numpy(),
            weights=(d.val[pos] * torch.repeat_interleave(d.w0[cols], cnt)).cpu().numpy(), minlength=d.n)).to(DEV)
        s.delta, s.phi = torch.empty_like(d.w0), torch.empty_like(d.w0)
        s.kkt = torch.empty(1, dtype=torch.float64, device=DEV)
    return s


def run(s):
    # "grad": the KKT violation is what max |g_j| has beyond lambda, a
    # difference that cancels near the optimum, so it is given with lambda
    case, kind = s.case, s.kind
    if kind == "run":  # warm start, iterations, their evaluation, w back on the device
        s.p.set_w(s.d.w0)
        s.p.set_iteration(0)
        r = s.p.iterate(case["iters"])
        return {"w": gb.gencd_get_w(s.p.h, s.d.k, s.w), "objective": r.objective, "grad": s.d.lam + r.kkt}
    if kind == "create":
        with _problem(case, s.d) as p:
            r = p.iterate(case["iters"])
            return {"w": p.w(), "objective": r.objective, "grad": s.d.lam + r.kkt}
    if kind == "path":
        recs, w, _ = s.b.path(s.held_out, s.lams, want_w=True)
        return {"w": w, "objective": np.array([x["objective"] for x in recs])}
    if kind == "noalloc":
        d = s.d
        gb.gencd_propose_all_noalloc(d.n, d.k, d.nnz, d.col_ptr, d.row_idx, d.val, d.y, s.z, d.w0, d.loss, d.lam, 0,
                                     s.delta, s.phi, s.kkt)
        return {"delta": s.delta, "phi": s.phi, "kkt": s.kkt}
    out, ws = gb.gencd_serve(s.problems, s.fracs, s.arrivals, workers=case["slots"], precision="f32",
                             hbm_fraction=0.05, want_w=True, variant="thread_greedy", blocks=case["blocks"],
                             max_iter=case["iters"], tol_kkt=0.0)
    return {"w": ws, "objective": np.array([r["objective"] for r in out])}


def work(case):
    """Bytes: every iteration reads the entries it proposes on (X stays in
    memory between iterations), and w is written once; flops: two per entry."""
    kind, k = case["kind"], case["k"]
    nnz = case["nnz"] if "nnz" in case else case["per_col"] * k
    size = {"f64": 12, "f32": 8, "bf16": 6, "binary": 4}[case.get("precision", "f64" if kind == "noalloc" else "f32")]
    if kind == "noalloc":
        return {"bytes": 12.0 * nnz + 16.0 * case["n"] + 32.0 * k, "flops": 4.0 * nnz}
    if kind == "path":  # the slots of a step share one read of X
        steps = case["iters"] * case["nlambda"]
        live = case["chains"]
        return {"bytes": 8.0 * nnz * steps + 8.0 * k * live * case["nlambda"], "flops": 2.0 * nnz * steps * live}
    if kind == "serve":
        entries = float(case["nreq"]) * case["iters"] * nnz
        return {"bytes": 8.0 * entries + 8.0 * k * case["nreq"], "flops": 2.0 * entries}
    per = float(nnz)
    if case["variant"] == "shotgun":
        per = float(nnz) * min(1.0, case["P"] / k)
    elif case["variant"] == "coloring":
        # a colour class is about n / (rows' largest degree) columns: k over
        # the number of colours, which is at least the mean degree
        per = float(nnz) / max(1.0, nnz / case["n"])
    first = nnz * size if kind == "create" else 0
    return {"bytes": per * size * (case["iters"] + 1) + first + 16.0 * k, "flops": 2.0 * per * (case["iters"] + 1)}


def tolerance(case):
    """FP64: sums in another order gave 4e-15 at most over repeats and against
    exact(), 4e-14 in the largest difference.  FP32 sums: up to 4e-7 in all and
    1e-6 in the largest difference for one to twenty iterations.  Where the
    best column of each of many partitions is taken in FP32 arithmetic, one
    choice in about 1e4 is between proxies that agree to their rounding
    (1e-6); the other choice moves another column, and w, objective and
    gradient of a correct run then differ by that one step, up to 6e-3 seen."""
    if case["kind"] == "noalloc" or case.get("precision") == "f64":
        return {"rel": 1e-12, "max": 1e-10}
    if case["kind"] in ("path", "serve") or case["variant"] in ("thread_greedy", "greedy"):
        return {"rel": 2e-2, "max": 0.99}
    return {"rel": 2e-6, "max": 1e-4}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch

class _Exact:
    def __init__(self, case, d, rows=None):
        self.n = d.n if rows is None else int(rows.sum())
        self.k, self.loss, self.lam, self.y = d.k, d.loss, d.lam, d.y
        self.col_ptr, self.row = d.col_ptr, d.row_idx.long()
        self.counts = d.col_ptr[1:] - d.col_ptr[:-1]
        v = d.val
        if case.get("precision") == "bf16":
            v = v.to(torch.bfloat16)
        self.val = v.double()
        self.rows = rows  # training rows (None: all)
        sq = self.val * self.val
        if rows is not None:
            sq = sq * rows[self.row]
        c = _segment_sums(sq, self.counts) / self.n
        self.beta = (1.0 if d.loss == "squared" else 0.25) * c
        # the narrowest relative gap so far between a partition's two best
        # proxies, and the one below which rounding decides which wins
        self.gap, self.tie = math.inf, 1e-12 if v.dtype == torch.float64 else 1e-5
        self.XT = torch.sparse_csr_tensor(self.col_ptr, self.row, self.val, size=(d.k, d.n))

    def u(self, z):
        u = z - self.y if self.loss == "squared" else -self.y * torch.sigmoid(-self.y * z)
        return u if self.rows is None else u * self.rows

    def fitted(self, w):
        z = torch.zeros_like(self.y)
        self.add(z, torch.nonzero(w).flatten(), w)
        return z

    def add(self, z, cols, d):
        pos, cnt = _entries_of(self.col_ptr, cols)
        z.index_add_(0, self.row[pos], self.val[pos] * torch.repeat_interleave(d[cols], cnt))

    def step(self, g, w, beta):
        lo, hi, t = g - self.lam, g + self.lam, w * beta
        safe = torch.where(beta > 0, beta, torch.ones_like(beta))
        d = torch.where(t < lo, -lo / safe, torch.where(t > hi, -hi / safe, -w))
        d = torch.where(beta > 0, d, -w)
        x = w + d
        keep = (w != 0) & ((torch.sign(w) == torch.sign(x)) | (x == 0))
        dabs = torch.where(keep, torch.sign(w) * d, x.abs() - w.abs())
        return d, torch.where(beta > 0, d * (0.5 * beta * d + g) + self.lam * dabs, -self.lam * w.abs())

    def propose(self, w, z):
        g = (self.XT @ self.u(z)) / self.n
        return (g,) + self.step(g, w, self.beta)

    def thread_greedy(self, w, z, B):
        _, d, f = self.propose(w, z)
        B = max(1, min(B, self.k))
        part = ((torch.arange(self.k, device=DEV) + 1) * B - 1) // self.k
        best = torch.zeros(B, dtype=torch.float64, device=DEV).scatter_reduce_(0, part, f, "amin")
        hit = torch.nonzero((f == best[part]) & (f < 0)).flatten()
        first = torch.full((B,), self.k, device=DEV).scatter_reduce_(0, part[hit], hit, "amin")
        f[first[first < self.k]] = 0.0
        second = torch.zeros(B, dtype=torch.float64, device=DEV).scatter_reduce_(0, part, f, "amin")
        gaps = ((second - best) / best.abs())[best < 0]
        gaps = gaps[gaps != 0]  # equal proxies: the lower column, at any precision
        if gaps.numel():
            self.gap = min(self.gap, float(gaps.min()))
        self.apply(w, z, first[first < self.k], d)

    def some(self, w, z, cols):
        """Every listed column's step from the present state."""
        pos, cnt = _entries_of(self.col_ptr, cols)
        g = _segment_sums(self.val[pos] * self.u(z)[self.row[pos]], cnt) / self.n
        d = torch.zeros_like(w)
        d[cols] = self.step(g, w[cols], self.beta[cols])[0]
        self.apply(w, z, cols, d)

    def apply(self, w, z, cols, d):
        w[cols] += d[cols]
        self.add(z, cols, d)

    def sure(self, w):
        """w, unless a choice on the way to it was a matter of rounding."""
        return w if self.gap > self.tie else None

    def evaluate(self, w, z):
        if self.loss == "squared":
            l = 0.5 * (self.y - z) ** 2
        else:
            m = -self.y * z
            l = torch.clamp(m, min=0) + torch.log1p(torch.exp(-m.abs()))
        if self.rows is not None:
            l = l * self.rows
        g = (self.XT @ self.u(z)) / self.n
        v = torch.where(w == 0, torch.clamp(g.abs() - self.lam, min=0), (g + self.lam * torch.sign(w)).abs())
        return float(l.sum() / self.n + self.lam * w.abs().sum()), float(v.max())


def _mix(x):
    with np.errstate(over="ignore"):
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return x ^ (x >> np.uint64(31))


def _permutation(epoch, m):
    """Select's order: 0..m-1 sorted by the top half of SplitMix64 outputs."""
    gamma = np.uint64(0x9E3779B97F4A7C15)
    with np.errstate(over="ignore"):
        s = _mix(np.uint64(0) + np.uint64(epoch + 1) * gamma)
        keys = _mix(s + (np.arange(m, dtype=np.uint64) + np.uint64(1)) * gamma) >> np.uint64(32)
    return np.argsort(keys, kind="stable")


def _first_fit(d):
    """Columns in order, each with the least colour none of its rows' columns has."""
    cp, row = d.col_ptr.cpu().numpy(), d.row_idx.cpu().numpy()
    used, colour = [0] * d.n, np.empty(d.k, np.int64)
    for j in range(d.k):
        rows, m = row[cp[j]:cp[j + 1]], 0
        for i in rows:
            m |= used[i]
        c = (~m & (m + 1)).bit_length() - 1
        colour[j] = c
        for i in rows:
            used[i] |= 1 << c
    return colour


def _iterate(case, d, e, w, z):
    v, iters = case["variant"], case["iters"]
    if v in ("thread_greedy", "greedy"):
        for _ in range(iters):
            e.thread_greedy(w, z, 1 if v == "greedy" else case["blocks"])
        return
    if v == "shotgun":
        P = min(case["P"], d.k)
        per = -(-d.k // P)
        for t in range(iters):
            if t % per == 0:
                perm = torch.from_numpy(_permutation(t // per, d.k)).to(DEV)
            e.some(w, z, perm[(t % per) * P:(t % per + 1) * P])
        return
    colour = _first_fit(d)
    classes = [torch.from_numpy(np.flatnonzero(colour == c)).to(DEV) for c in range(int(colour.max()) + 1)]
    for t in range(iters):
        if t % len(classes) == 0:
            perm = _permutation(t // len(classes), len(classes))
        e.some(w, z, classes[int(perm[t % len(classes)])])


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        ws, obj = [], []
        for q, r in enumerate(_requests(case, seed)):
            d = types.SimpleNamespace(n=r.n, k=r.k, loss=r.loss, col_ptr=torch.from_numpy(r.col_ptr).to(DEV),
                                      row_idx=torch.from_numpy(r.row_idx).to(DEV),
                                      val=torch.from_numpy(r.val).to(DEV), y=torch.from_numpy(r.y).to(DEV), lam=0.0)
            e = _Exact(case, d)
            e.lam = case["lam"] * float((e.XT @ e.u(torch.zeros_like(e.y))).abs().max()) / d.n
            w, z = torch.zeros(d.k, dtype=torch.float64, device=DEV), torch.zeros_like(d.y)
            for _ in range(case["iters"]):
                e.thread_greedy(w, z, case["blocks"])
            ws.append(e.sure(w))
            obj.append(e.evaluate(w, z)[0])
        return {"w": ws, "objective": np.array(obj)}
    d = _data(case, seed)
    if kind == "path":
        held_out, lams = _path_grid(case, d)
        fold = _fold(case)
        W, obj = [], []
        sets = [_Exact(case, d, (fold != f).double()) for f in range(case["folds"])]
        for c in range(case["chains"]):
            e = sets[int(held_out[c])]
            w, z = torch.zeros(d.k, dtype=torch.float64, device=DEV), torch.zeros_like(d.y)
            for lam in lams[c]:
                e.lam = float(lam)
                for _ in range(case["iters"]):
                    e.thread_greedy(w, z, case["blocks"])
                W.append(w.cpu().numpy().copy())
                obj.append(e.evaluate(w, z)[0])
        sure = all(e.gap > e.tie for e in sets)
        return {"w": np.array(W).reshape(case["chains"], case["nlambda"], d.k) if sure else None,
                "objective": np.array(obj)}
    e = _Exact(case, d)
    w = d.w0.clone() if kind != "create" else torch.zeros_like(d.w0)
    z = e.fitted(w)
    if kind == "noalloc":
        g, dl, f = e.propose(w, z)
        return {"delta": dl, "phi": f, "kkt": torch.tensor([e.evaluate(w, z)[1]], dtype=torch.float64)}
    _iterate(case, d, e, w, z)
    objective, kkt = e.evaluate(w, z)
    return {"w": e.sure(w if kind != "create" else w.cpu().numpy()), "objective": objective, "grad": d.lam + kkt}
