"""Initialisation at the edges of the radix sort's tiles (2,048 records up to 2^19 nonzeros, 8,192
above): with rank 1 and factors of ones, Y_(n) holds the sums of the slices' values, which are small
integers, so they are exact in any order and equal numpy's."""
import numpy as np
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz", [1, 2047, 2048, 2049, 16_385, 100_003, 2**19, 2**19 + 1, 2**19 + 8193])
def test_slice_sums(nnz):
    T = lib()
    dims = (700, 300, 1100)
    rng = np.random.default_rng(nnz)
    coords = np.stack([np.minimum(rng.geometric(0.01, nnz) - 1, dims[0] - 1), rng.integers(0, dims[1], nnz),
                       rng.integers(0, dims[2], nnz)]).astype(np.int32)
    vals = rng.integers(-8, 9, nnz).astype(np.float32)
    ctx = T.tucker_init(dims, torch.as_tensor(coords).cuda(), torch.as_tensor(vals).cuda(), (1, 1, 1),
                        [torch.ones(d, 1, dtype=torch.float64, device="cuda") for d in dims])
    for n in range(3):
        want = np.bincount(coords[n], weights=vals, minlength=dims[n])
        np.testing.assert_array_equal(T.ttmc_mode(ctx, n).cpu().numpy()[:, 0], want)
    T.tucker_free(ctx)
