"""The loss of tucker_loss_grad at the ends of FP32's range: with the values and the core scaled by 2^p,
every residual is scaled by 2^p, and the loss, a sum of their squares in FP64, by 4^p, whether or not the
squares fit in FP32.  (The gradients of the factors are products of two scaled numbers and leave FP32's
range by themselves; those of the core are scaled by 2^p.)

Bar: 1e-6.  Up, every FP32 operation scales exactly.  Down, products of the model that fall below 2^-126
lose up to 2^-149 each, 2^-58 of a residual in all, which may turn a rounding of the residual: 2^-23 of
it, and twice that of its square.

Shapes: the fused form at orders 2 to 5 (padded tiles, several groups, slices cut over many units), and
one it does not cover."""
import zlib

import numpy as np
import pytest

from tests.gpu_util import lib, rel_fro, torch

pytestmark = pytest.mark.gpu

CASES = [
    ((200, 64), (5, 17), 4000),
    ((60, 50, 40), (10, 10, 10), 6000),
    ((3, 64, 60), (3, 16, 16), 5000),
    ((30, 20, 25, 22), (3, 5, 5, 5), 4000),
    ((12, 10, 11, 9, 8), (2, 3, 3, 3, 3), 3000),
    ((40, 70, 80), (2, 40, 64), 3000),  # 64 tiles and more: not covered
]


@pytest.mark.parametrize("power", [70, -80])
@pytest.mark.parametrize("dims,ranks,nnz", CASES, ids=["x".join(map(str, c[1])) for c in CASES])
def test_loss_scales(dims, ranks, nnz, power):
    T = lib()
    rng = np.random.default_rng(zlib.crc32(repr(ranks).encode()))
    flat = rng.choice(int(np.prod(dims)), size=nnz, replace=False)
    coords = torch.as_tensor(np.stack(np.unravel_index(flat, dims)).astype(np.int32)).cuda()
    vals = torch.as_tensor(rng.standard_normal(nnz).astype(np.float32)).cuda()
    U = [torch.as_tensor(rng.standard_normal((d, r)).astype(np.float32)).cuda() for d, r in zip(dims, ranks)]
    G = torch.as_tensor((rng.standard_normal(ranks) / np.sqrt(np.prod(ranks))).astype(np.float32)).cuda()
    out = []
    for s in (1.0, 2.0**power):
        ctx = T.tucker_init(dims, coords, vals * s, ranks, seed=1)
        L, _, dG = T.tucker_loss_grad(ctx, U, G * s)
        out.append((float(L), dG.double().cpu().numpy() / s))
        T.tucker_free(ctx)
    assert out[1][0] / 4.0**power == pytest.approx(out[0][0], rel=1e-6)
    assert rel_fro(out[1][1], out[0][1]) <= 1e-6
