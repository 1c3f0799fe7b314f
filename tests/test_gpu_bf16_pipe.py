"""BF16 contexts of order 3 whose ranks the tensor-core form does not cover but the FP32 pipeline does: the
same kernel as in an FP32 context that was given the BF16-rounded factors, so the same bits; without the
pipeline (unpipelined) the tiled form, within the bound of sums of the same products in another order."""
import numpy as np
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ranks,modes", [((8, 8, 8), (0, 1, 2)), ((8, 16, 8), (1, 2)), ((16, 8, 16), (0,))],
                         ids=["8x8x8", "8x16x8", "16x8x16"])
@pytest.mark.parametrize("chunk", [None, 32])
def test_same_as_fp32_on_rounded_factors(ranks, modes, chunk, monkeypatch):
    T = lib()
    monkeypatch.setenv("TUCKER_TTMC_FIBERS", "0")
    if chunk:
        monkeypatch.setenv("TUCKER_TTMC_CHUNK", str(chunk))
    rng = np.random.default_rng(sum(ranks))
    dims, n = (70, 60, 50), 20_011
    coords = torch.as_tensor(np.stack([rng.integers(0, d, n) for d in dims]).astype(np.int32)).cuda()
    vals = torch.as_tensor(rng.standard_normal(n).astype(np.float32)).cuda()
    U = [torch.as_tensor(rng.standard_normal((d, r))).cuda() for d, r in zip(dims, ranks)]
    bf = T.tucker_init(dims, coords, vals, ranks, U, bf16=True)
    fp = T.tucker_init(dims, coords, vals, ranks, [u.bfloat16().double() for u in U])
    plain = T.tucker_init(dims, coords, vals, ranks, U, bf16=True, unpipelined=True)
    for m in modes:
        Y = T.ttmc_mode(bf, m)
        assert torch.equal(Y, T.ttmc_mode(fp, m)), m
        a = torch.linalg.norm(T.ttmc_mode(plain, m).double() - Y.double()) / torch.linalg.norm(Y.double())
        assert 0 < float(a) <= 1e-5, m
