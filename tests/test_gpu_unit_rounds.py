"""Work units of the BF16 form of order 4, of which an SM holds few: half as long where that leaves a last
round less empty, and the same Y to the BF16 form's rounding of its products."""
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz,chunk", [(300_000, 128), (450_000, 128), (500_000, 256), (1_000_000, 128), (2_000_000, 256)])
def test_chunk(nnz, chunk):
    """152 SMs hold 3,648 units: 2 x 256 or 3 x 128 nonzeros of a slot at 1M, 256 either way at 500,000."""
    T = lib()
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("numbers for 152 SMs")
    g = torch.Generator(device="cuda").manual_seed(1)
    dims, ranks = (200,) * 4, (8,) * 4
    coords = torch.stack([torch.randint(0, d, (nnz,), generator=g, device="cuda", dtype=torch.int32) for d in dims])
    vals = torch.randn(nnz, generator=g, device="cuda")
    U = [torch.randn((d, r), generator=g, device="cuda", dtype=torch.float64) for d, r in zip(dims, ranks)]
    bf = T.tucker_init(dims, coords, vals, ranks, U, bf16=True)
    fp = T.tucker_init(dims, coords, vals, ranks, [u.bfloat16().double() for u in U])
    assert T.tucker_mode_info(bf, 0)["chunk"] == chunk
    assert T.tucker_mode_info(fp, 0)["chunk"] == (256 if nnz >= 400_000 else 128)
    Y, want = T.ttmc_mode(bf, 0).double(), T.ttmc_mode(fp, 0).double()
    assert float(torch.linalg.norm(Y - want) / torch.linalg.norm(want)) <= 1e-2
