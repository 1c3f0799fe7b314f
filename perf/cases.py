"""What the speed of this framework is measured on: calls that its users make, through its
public entry points (paper_2010_10638_gb300.tucker and .autograd).

Kinds of case (`kind`):

  ttmc   the sparse tensor-times-matrix chain of every mode (ttmc_mode), on a loaded tensor:
         the step of a sweep that grows with the nonzeros, also called by itself (sketches,
         custom sweeps).  FP32 factors, or BF16 copies (`bf16`).
  qrp    QR with column pivoting of an FP64 matrix (qrp_leading): Q, pivots, diag(R).
  grad   one training step of a completion model on the observed entries: the loss and the
         gradients of every factor and of the core (tucker_loss, autograd).
  sweep  one HOOI sweep (hooi_iter) from given factors; the core and the factors are then
         handed on in FP32, the form in which the training step above takes a model.
  load   a tensor that has just arrived on the GPU as COO: tucker_init, `sweeps` HOOI sweeps,
         the core and the factors as for `sweep`, and the release of the context.

Sizes are those of the workload recipes (paper_2010_10638_gb300/synth.py), of the tests and
of the benchmark.  Inputs are drawn on the GPU from the seed.
"""
import math

import torch

from paper_2010_10638_gb300 import tucker as T
from paper_2010_10638_gb300.autograd import tucker_loss


def listed():
    return [
        # the smallest call: a 100^3 tensor, where launches and latency are all there is
        dict(name="ttmc-tiny", kind="ttmc", dims="100x100x100", ranks="8x8x8", nnz=10_000, coords="uniform",
             values="uniform", bf16=False),
        # ranks that follow the data and sizes that divide nothing
        dict(name="ttmc-ragged", kind="ttmc", dims="2003x1501x907", ranks="12x7x20", nnz=600_011, coords="zipf",
             values="normal", bf16=False),
        # the benchmark's tensor: 20M nonzeros, one skewed mode, FP32 factors
        dict(name="ttmc-skew-20m", kind="ttmc", dims="50000x50000x1000", ranks="16x16x16", nnz=20_000_000,
             coords="skew", values="lognormal", bf16=False),
        # the same tensor with BF16 copies of the factors, the option for speed
        dict(name="ttmc-skew-20m-bf16", kind="ttmc", dims="50000x50000x1000", ranks="16x16x16", nnz=20_000_000,
             coords="skew", values="lognormal", bf16=True),
        # an order-4 tensor
        dict(name="ttmc-order4-5m", kind="ttmc", dims="5000x5000x2000x500", ranks="8x8x8x8", nnz=5_000_000,
             coords="uniform", values="normal", bf16=False),
        # a tall FP64 matrix factored by itself
        dict(name="qrp-tall", kind="qrp", rows=20_000, cols=256, k=16),
        # one training step: a small model, and the completion workload
        dict(name="grad-small", kind="grad", dims="200x150x100", ranks="8x8x8", nnz=50_000),
        dict(name="grad-completion-10m", kind="grad", dims="20000x20000x20000", ranks="10x10x10", nnz=10_000_000),
        # one sweep: a 200^3 tensor (every unfolding fat: the Gram branch), an order-4 tensor, the benchmark's step
        dict(name="sweep-200", kind="sweep", dims="200x200x200", ranks="16x16x16", nnz=80_000, coords="uniform",
             values="normal"),
        dict(name="sweep-skew-20m", kind="sweep", dims="50000x50000x1000", ranks="16x16x16", nnz=20_000_000,
             coords="skew", values="lognormal"),
        # a whole job on a new tensor of 1M skewed nonzeros
        dict(name="load-zipf-1m", kind="load", dims="10000x10000x10000", ranks="16x16x16", nnz=1_000_000,
             coords="zipf", values="normal", sweeps=2),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ranks(rng, order):
    """Ranks of one tensor: a power of two in every mode, one odd number in every mode, or one for each."""
    top = {2: 32, 3: 32, 4: 9, 5: 5}[order]
    how = rng.randrange(3)
    if how == 0:
        r = [rng.choice([v for v in (4, 8, 16, 32) if v <= top])] * order
    elif how == 1:
        r = [rng.randint(3, top)] * order
    else:
        r = [rng.randint(3, top) for _ in range(order)]
    return r


def _spell(v):
    return "x".join(str(int(x)) for x in v)


def draw(rng):
    """One more case of the same kinds: orders 2 to 5, ranks 3 to 32, 10,000 to 10M nonzeros."""
    kind = rng.choice(["ttmc", "ttmc", "ttmc", "grad", "grad", "sweep", "qrp", "load"])
    if kind == "qrp":
        k = rng.choice([8, 10, 12, 16, 16, 24])
        rows = _loguniform(rng, 200, 40_000)
        return dict(kind="qrp", rows=rows, cols=rng.randint(k, 256), k=k)
    order = rng.choice([3, 3, 3, 4]) if kind in ("sweep", "load") else rng.choice([2, 3, 3, 3, 3, 4, 5])
    ranks = _ranks(rng, order)
    if kind in ("sweep", "load"):  # R_n <= the columns of Y_(n)
        ranks = [min(r, 16) for r in ranks] if order == 3 else [min(r, 8) for r in ranks]
        ranks = [min(r, math.prod(ranks) // r) for r in ranks]
    cells = math.prod(ranks) // min(ranks)  # columns of the widest Y_(n)
    most = min(10_000_000, 2_500_000_000 // (cells * order))
    nnz = _loguniform(rng, 10_000, max(20_000, most))
    dims = [max(_loguniform(rng, 40, 30_000), 2 * r) for r in ranks]
    while math.prod(dims) < 8 * nnz:  # the tensor stays sparse
        dims = [d * 2 + 1 for d in dims]
    while max(d * math.prod(ranks) // r for d, r in zip(dims, ranks)) > 100_000_000:  # 400 MB of Y_(n) at most
        dims = [max(d // 2, 2 * r) for d, r in zip(dims, ranks)]
    c = dict(kind=kind, dims=_spell(dims), ranks=_spell(ranks), nnz=nnz)
    if kind != "grad":
        c["coords"] = rng.choice(["uniform", "zipf", "skew"])
        c["values"] = "normal" if kind in ("sweep", "load") else rng.choice(["normal", "uniform", "lognormal"])
    if kind == "ttmc":
        c["bf16"] = rng.random() < 0.25
    if kind == "load":
        c["sweeps"] = 1
    return c


# ------------------------------------------------------------------------------------ inputs
def _list(text):
    return [int(x) for x in text.split("x")]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, size, nnz):
    return torch.randint(0, size, (nnz,), generator=g, device="cuda", dtype=torch.int32)


def _zipf(g, size, nnz, s):
    """P(i) ~ (i + 1)^-s on [0, size), then a random relabelling."""
    cdf = torch.cumsum(torch.arange(1, size + 1, device="cuda", dtype=torch.float64) ** -s, 0)
    u = torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    rank = torch.searchsorted(cdf, u).clamp_(max=size - 1)
    return torch.randperm(size, generator=g, device="cuda")[rank].to(torch.int32)


def _coords(g, how, dims, nnz):
    if how == "uniform":
        c = [_uniform(g, d, nnz) for d in dims]
    elif how == "zipf":
        c = [_zipf(g, d, nnz, 1.1) for d in dims]
    else:  # "skew": the first mode only
        c = [_zipf(g, dims[0], nnz, 1.2)] + [_uniform(g, d, nnz) for d in dims[1:]]
    return torch.stack(c)


def _values(g, how, nnz):
    if how == "uniform":
        return torch.rand(nnz, generator=g, device="cuda")
    v = torch.randn(nnz, generator=g, device="cuda")
    return v.exp_() if how == "lognormal" else v


def _orthonormal(g, rows, cols):
    q, _ = torch.linalg.qr(torch.randn((rows, cols), generator=g, device="cuda", dtype=torch.float64))
    return q.contiguous()


def _tensor(case, seed):
    """COO and initial factors (the kinds ttmc, sweep and load)."""
    g = _gen(seed)
    dims, ranks = _list(case["dims"]), _list(case["ranks"])
    coords = _coords(g, case["coords"], dims, case["nnz"])
    vals = _values(g, case["values"], case["nnz"])
    return dims, ranks, coords, vals, [_orthonormal(g, d, r) for d, r in zip(dims, ranks)]


def _completion(case, seed):
    """Observed entries of a Tucker model plus noise, and the model that is being trained: the
    generating one, perturbed."""
    g = _gen(seed)
    dims, ranks = _list(case["dims"]), _list(case["ranks"])
    coords = _coords(g, "uniform", dims, case["nnz"])
    U = [torch.randn((d, r), generator=g, device="cuda") for d, r in zip(dims, ranks)]
    G = torch.randn(ranks, generator=g, device="cuda") / math.sqrt(math.prod(ranks))
    vals = _model_values(coords, U, G) + 0.01 * torch.randn(case["nnz"], generator=g, device="cuda")
    U = [u + 0.1 * torch.randn(u.shape, generator=g, device="cuda") for u in U]
    return dims, ranks, coords, vals, U, G


def _model_values(coords, U, G, chunk=1 << 20):
    """sum_r G[r] prod_m U_m(i_m, r_m) at each coordinate, in the type of U and G."""
    out = []
    for s in range(0, coords.shape[1], chunk):
        c = coords[:, s:s + chunk].long()
        acc = (U[0] @ G.reshape(G.shape[0], -1))[c[0]] if U[0].shape[0] < c.shape[1] else U[0][c[0]] @ G.reshape(G.shape[0], -1)
        for m in range(1, len(U)):
            acc = torch.bmm(U[m][c[m]].unsqueeze(1), acc.reshape(c.shape[1], U[m].shape[1], -1)).squeeze(1)
        out.append(acc.reshape(-1))
    return torch.cat(out)


# ------------------------------------------------------------------------------------ the cases
class State:
    pass


def prepare(case, seed):
    T.load()
    s = State()
    s.kind = case["kind"]
    if s.kind == "qrp":
        g = _gen(seed)
        s.k = case["k"]
        s.A = torch.randn((case["rows"], case["cols"]), generator=g, device="cuda", dtype=torch.float64)
        s.A *= 0.2 + 4.8 * torch.rand(case["cols"], generator=g, device="cuda", dtype=torch.float64)
        s.work = torch.empty(T.qrp_leading_work_bytes(*s.A.shape, s.k), dtype=torch.uint8, device="cuda")
        return s
    if s.kind == "grad":
        s.dims, s.ranks, coords, vals, U, G = _completion(case, seed)
        s.ctx = T.tucker_init(s.dims, coords, vals, s.ranks, seed=1)
        s.U = [u.requires_grad_(True) for u in U]
        s.G = G.requires_grad_(True)
        return s
    s.dims, s.ranks, coords, vals, s.U0 = _tensor(case, seed)
    if s.kind == "load":
        s.coords, s.vals, s.sweeps = coords, vals, case["sweeps"]
        return s
    s.ctx = T.tucker_init(s.dims, coords, vals, s.ranks, s.U0, bf16=case.get("bf16", False))
    if s.kind == "ttmc":
        s.Y = [torch.empty((d, s.ctx.P(n)), device="cuda") for n, d in enumerate(s.dims)]
    return s


def _model(ctx):
    """The decomposition as an FP32 model (core and factors), as tucker_loss_grad takes it."""
    return [T.core_tensor(ctx).float()] + [T.tucker_get_factor(ctx, n).float() for n in range(ctx.N)]


def run(s):
    if s.kind == "qrp":
        return T.qrp_leading(s.A, s.k, work=s.work)
    if s.kind == "ttmc":
        for n in range(len(s.dims)):
            T.ttmc_mode(s.ctx, n, s.Y[n])
        return s.Y
    if s.kind == "grad":
        loss = tucker_loss(s.ctx, s.G, s.U).float()  # joined with the FP32 terms of an objective
        return [loss.detach(), *torch.autograd.grad(loss, [s.G, *s.U])]
    if s.kind == "sweep":
        for n in range(1, len(s.dims)):  # a sweep reads the factors of modes 2 .. N
            T.tucker_set_factor(s.ctx, n, s.U0[n])
        fit = T.hooi_iter(s.ctx)
        return [fit, *_model(s.ctx)]
    ctx = T.tucker_init(s.dims, s.coords, s.vals, s.ranks, s.U0)
    for _ in range(s.sweeps):
        fit = T.hooi_iter(ctx)
    out = [fit, *_model(ctx)]
    T.tucker_free(ctx)
    return out


def work(case):
    """Each input read once, each output written once; the additions and multiplications of the method."""
    if case["kind"] == "qrp":
        m, n, k = case["rows"], case["cols"], case["k"]
        return {"bytes": 8 * (m * n + m * k + 2 * k), "flops": 4 * m * n * k + 4 * m * k * k}
    dims, ranks, nnz = _list(case["dims"]), _list(case["ranks"]), case["nnz"]
    N, core = len(dims), math.prod(ranks)
    coo = 4 * (N + 1) * nnz
    ttmc = sum(2 * nnz * core // r for r in ranks)
    if case["kind"] == "ttmc":
        size = 2 if case["bf16"] else 4
        fac = sum(size * d * r for d, r in zip(dims, ranks))
        return {"bytes": N * (coo + fac) + sum(4 * d * core // r for d, r in zip(dims, ranks)), "flops": ttmc}
    if case["kind"] == "grad":
        model = 4 * (core + sum(d * r for d, r in zip(dims, ranks)))
        return {"bytes": (N + 1) * coo + 2 * model, "flops": ttmc + 2 * nnz * core // ranks[0] + 4 * sum(d * core for d in dims)}
    sweeps = case.get("sweeps", 1)
    Y = [4 * d * core // r for d, r in zip(dims, ranks)]
    model = 12 * (core + sum(d * r for d, r in zip(dims, ranks)))
    qrp = sum(4 * min(y // 4, d * d) * r for y, d, r in zip(Y, dims, ranks))
    return {"bytes": sweeps * (N * coo + 2 * sum(Y)) + (3 * N * coo if case["kind"] == "load" else 0) + model,
            "flops": sweeps * (ttmc + qrp + 2 * dims[-1] * core)}


# ------------------------------------------------------------------------------------ in 64 bits
def _coalesced(coords, vals, dims):
    key = torch.zeros(coords.shape[1], dtype=torch.int64, device="cuda")
    for c, d in zip(coords, dims):
        key = key * d + c
    key, back = torch.unique(key, return_inverse=True)
    v = torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, back, vals.double())
    out = []
    for d in reversed(dims):
        out.append(key % d)
        key = torch.div(key, d, rounding_mode="floor")
    return torch.stack(out[::-1]), v


class _Chain:
    """Y_(n) in 64 bits: for every column of the Kronecker product of all remaining modes but the
    last, a sparse matrix (rows i_n, columns i_last) times the last mode's factor."""

    def __init__(self, dims, coords, vals):
        self.dims, self.c, self.v = dims, coords.long(), vals.double()

    def __call__(self, n, U, v=None):
        v = self.v if v is None else v
        left = [m for m in range(len(U)) if m != n]
        last = left.pop()
        order = torch.argsort(self.c[n])
        rows = torch.zeros(self.dims[n] + 1, dtype=torch.int64, device="cuda")
        rows[1:] = torch.cumsum(torch.bincount(self.c[n], minlength=self.dims[n]), 0)
        cols, v = self.c[last][order], v[order]
        idx = [self.c[m][order] for m in left]
        L = math.prod(U[m].shape[1] for m in left)
        Y = torch.empty((self.dims[n], L, U[last].shape[1]), dtype=torch.float64, device="cuda")
        for j in range(L):
            w, q = v, j
            for m, i in zip(reversed(left), reversed(idx)):
                q, r = divmod(q, U[m].shape[1])
                w = w * U[m][:, r][i]
            Y[:, j] = self._times(rows, cols, w, U[last])
        return Y.reshape(self.dims[n], -1)

    @staticmethod
    def _times(rows, cols, w, B):
        # a CSR matrix may not hold more entries than it has cells: repeated cells go in several matrices
        most, out = (rows.numel() - 1) * B.shape[0], 0
        for s in range(0, cols.numel(), most):
            n = min(most, cols.numel() - s)
            out = out + torch.sparse_csr_tensor((rows - s).clamp(0, n), cols[s:s + n], w[s:s + n],
                                                size=(rows.numel() - 1, B.shape[0])) @ B
        return out


def _qrp(A, k):
    """k Householder reflectors with column pivoting: Q, pivots, diagonal of R."""
    A = A.clone()
    m, n = A.shape
    perm = torch.arange(n, device="cuda")
    V, beta = [], []
    for j in range(k):
        p = j + int(torch.argmax((A[j:, j:] ** 2).sum(0)))
        A[:, [j, p]] = A[:, [p, j]]
        perm[[j, p]] = perm[[p, j]]
        v = A[j:, j].clone()
        alpha = torch.linalg.norm(v) * (-1.0 if float(v[0]) < 0 else 1.0)
        v[0] += alpha
        w = 2.0 / torch.dot(v, v)
        A[j:, j:] -= torch.outer(w * v, v @ A[j:, j:])
        V.append((v, w))
        beta.append(-alpha)
    Q = torch.zeros((m, k), dtype=torch.float64, device="cuda")
    Q[range(k), range(k)] = 1.0
    for j in reversed(range(k)):
        v, w = V[j]
        Q[j:] -= torch.outer(w * v, v @ Q[j:])
    return Q, perm[:k].clone(), torch.stack(beta)


def _sweeps(case, seed):
    dims, ranks, coords, vals, U = _tensor(case, seed)
    coords, v = _coalesced(coords, vals, dims)
    chain, norm2 = _Chain(dims, coords, v), float((v * v).sum())
    for _ in range(case.get("sweeps", 1)):
        for n in range(len(dims)):
            Y = chain(n, U)
            U[n] = _qrp(Y @ Y.T if Y.shape[1] > Y.shape[0] else Y, ranks[n])[0]
    G = (Y.T @ U[-1]).reshape(*ranks)
    fit = 1.0 - math.sqrt(max(0.0, norm2 - float((G * G).sum()))) / math.sqrt(norm2)
    return [fit, G, *U]


def exact(case, seed):
    if case["kind"] == "qrp":
        s = prepare(case, seed)
        return _qrp(s.A, s.k)
    if case["kind"] == "ttmc":
        dims, ranks, coords, vals, U = _tensor(case, seed)
        chain = _Chain(dims, coords, vals)
        return [chain(n, U) for n in range(len(dims))]
    if case["kind"] in ("sweep", "load"):
        return _sweeps(case, seed)
    dims, ranks, coords, vals, U, G = _completion(case, seed)
    coords, v = _coalesced(coords, vals, dims)
    v = v.float().double()  # duplicates are summed into one FP32 observation
    U, G = [u.detach().double() for u in U], G.double()
    e = _model_values(coords, U, G) - v
    chain = _Chain(dims, coords, e)
    N, dU = len(dims), []
    for n in range(N):
        Y = chain(n, U)
        Gn = G.movedim(n, 0).reshape(ranks[n], -1)
        dU.append(Y @ Gn.T)
        if n == 0:
            dG = (U[0].T @ Y).reshape(*ranks)
    return [0.5 * float((e * e).sum()), dG, *dU]
