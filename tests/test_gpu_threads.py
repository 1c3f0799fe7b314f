"""Distinct contexts are independent: calls on two contexts from two host threads, each on its own stream,
that launch the same kernels with shared memory of different sizes (other ranks, the same tile), all
succeed and give what the same call gives by itself, bit for bit."""
import threading

import numpy as np
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu
DIMS = (300, 300, 300)


def context(T, ranks, nnz=120_000):
    rng = np.random.default_rng(sum(ranks))
    coords = np.stack([rng.integers(0, d, nnz) for d in DIMS]).astype(np.int32)
    vals = rng.standard_normal(nnz).astype(np.float32)
    return T.tucker_init(DIMS, torch.as_tensor(coords).cuda(), torch.as_tensor(vals).cuda(), ranks, seed=3)


def calls(T, ctx, kind, stream):
    """A function that makes one call, and the tensors it writes."""
    if kind == "ttmc":
        Y = torch.empty((DIMS[0], ctx.P(0)), device="cuda")
        return lambda: T.ttmc_mode(ctx, 0, Y, stream=stream), [Y]
    g = torch.Generator(device="cuda").manual_seed(1)
    U = [torch.randn((d, r), generator=g, device="cuda") for d, r in zip(DIMS, ctx.ranks)]
    G = torch.randn(ctx.ranks, generator=g, device="cuda")
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    dU, dG = [torch.empty_like(u) for u in U], torch.empty_like(G)
    return lambda: T.tucker_loss_grad(ctx, U, G, loss, dU, dG, stream=stream), [loss, dG, *dU]


@pytest.mark.parametrize("kind,ranks,n", [
    ("ttmc", [(10, 10, 20), (10, 10, 10)], 3000),  # tiles of 5 x 5, records of 48 and 32 floats
    ("grad", [(24, 24, 24), (10, 10, 10)], 1000),  # the contraction with G_(n): 78 and 5 KB
])
def test_two_threads(kind, ranks, n):
    T = lib()
    work, want = [], []
    for r in ranks:
        stream = torch.cuda.Stream()
        ctx = context(T, r)
        torch.cuda.synchronize()
        call, out = calls(T, ctx, kind, stream)
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        want.append([o.clone() for o in out])
        for o in out:
            o.zero_()
        work.append((call, out, stream))
    torch.cuda.synchronize()
    failed = []

    def go(call, stream):
        try:
            for i in range(n):
                call()
                if i % 100 == 99:
                    stream.synchronize()
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            failed.append(repr(e))

    threads = [threading.Thread(target=go, args=(c, s)) for c, _, s in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for (_, out, _), w in zip(work, want):
        assert all(torch.equal(a, b) for a, b in zip(out, w))


def test_one_graph_of_several_sizes():
    """The modes of one sweep run the same tile (5 x 5) with records of 48, 40 and 24 floats."""
    T = lib()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a, b = context(T, (5, 10, 20)), context(T, (5, 10, 20))
        fits = [T.hooi_iter(a, stream=stream) for _ in range(3)]
        fit = torch.zeros(1, dtype=torch.float64, device="cuda")
        for f in fits:
            T.tucker_hooi_graph(b, 1, fit, stream=stream)
            stream.synchronize()
            assert float(fit) == f
        for n in range(3):
            assert torch.equal(T.tucker_get_factor(a, n), T.tucker_get_factor(b, n))
