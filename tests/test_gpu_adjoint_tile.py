"""The adjoint's fused kernel (residuals, loss and mode 1's TTMc in one pass) against the FP64
oracle: every order, tiles that pad, groups that are not a power of two, mode-1 slices of one
nonzero and slices cut over many units, and shapes it does not cover (rows of more tiles than a
warp has lanes), which run one thread per nonzero.

Bar: FP32 sums over k terms, 1e-4 relative as in test_gpu_adjoint.py, with entries of magnitude 1.
"""
import zlib

import numpy as np
import pytest

import oracle
from gpu_util import lib, rel_fro

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # dims, ranks, observations, nonzeros per work unit (None: chosen)
    ((60, 50, 40), (10, 10, 10), 6000, None),
    ((3, 70, 60), (3, 13, 7), 5000, 32),
    ((3000, 50, 40), (8, 8, 8), 3100, None),
    ((50, 40, 45), (16, 16, 16), 5000, 32),
    ((50, 40, 60), (4, 24, 33), 4000, None),       # 24 x 33: 4 x 8 tiles
    ((40, 70, 80), (2, 40, 64), 3000, None),       # 64 tiles and more: not covered
    ((30, 20, 25, 22), (3, 5, 5, 5), 4000, None),  # 5 tiles of a group of 8
    ((30, 20, 25, 22), (4, 8, 8, 8), 4000, 64),
    ((12, 10, 11, 9, 8), (2, 3, 3, 3, 3), 3000, None),
    ((200, 64), (5, 17), 4000, None),
]


@pytest.mark.parametrize("dims,ranks,nnz,chunk", CASES, ids=["x".join(map(str, c[1])) for c in CASES])
def test_loss_grad(dims, ranks, nnz, chunk, monkeypatch):
    T = lib()
    if chunk:
        monkeypatch.setenv("TUCKER_TTMC_CHUNK", str(chunk))
    rng = np.random.default_rng(zlib.crc32(repr((dims, ranks)).encode()))
    flat = rng.choice(int(np.prod(dims)), size=nnz, replace=False)
    coords = np.stack(np.unravel_index(flat, dims)).astype(np.uint32)
    vals = rng.standard_normal(nnz).astype(np.float32)
    U = [rng.standard_normal((d, r)).astype(np.float32) for d, r in zip(dims, ranks)]
    G = (rng.standard_normal(ranks) / np.sqrt(np.prod(ranks))).astype(np.float32)
    ctx = T.tucker_init(dims, torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        seed=1)
    args = [torch.as_tensor(u).cuda() for u in U], torch.as_tensor(G).cuda()
    L, dU, dG = T.tucker_loss_grad(ctx, *args)
    Lr, dUr, dGr = oracle.loss_grad(dims, ranks, coords, vals.astype(np.float64), [u.astype(np.float64) for u in U],
                                    G.astype(np.float64))
    assert abs(float(L) - Lr) <= 1e-4 * abs(Lr)
    assert rel_fro(dG.cpu().numpy(), dGr) <= 1e-4
    for n in range(len(dims)):
        assert rel_fro(dU[n].cpu().numpy(), dUr[n]) <= 1e-4, n
    L2, dU2, dG2 = T.tucker_loss_grad(ctx, *args)
    assert torch.equal(L, L2) and torch.equal(dG, dG2) and all(torch.equal(a, b) for a, b in zip(dU, dU2))
