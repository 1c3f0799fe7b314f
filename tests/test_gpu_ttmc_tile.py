"""The tiled TTMc (any order, any ranks) against the FP64 oracle, at the edges of its tiles:
every chunk width, ranks that pad, ranks above 32, one to seven remaining modes, rows wider than
a warp's tiles, slices of one nonzero and slices cut over many units; BF16 contexts whose ranks
the tensor-core form does not cover; factors given to the adjoint at odd addresses.

Bar: |Y - Y*| <= (D + N) 2^-24 (|X| x_m |U_m|^T) per entry, the first-order bound of a sum
evaluated in a tree of depth D (lane sums of at most min(k_i, chunk) terms, 31 group sums, the
fixup over pieces of a cut slice) over products of N roundings.
"""
import zlib

import numpy as np
import pytest

import oracle
from gpu_util import f32_round, lib
from paper_2010_10638_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # dims, ranks, nonzeros, nonzeros per work unit (None: chosen)
    ((50, 40, 30), (5, 6, 7), 3001, None),
    ((40, 45, 50), (9, 13, 11), 4000, 32),
    ((60, 40, 50), (15, 17, 3), 5003, None),
    ((70, 30, 64), (1, 24, 33), 3000, None),
    ((2, 900, 700), (2, 20, 14), 20_000, 64),       # two slices, cut into hundreds of units
    ((9000, 40, 50), (8, 10, 12), 5000, None),      # slices of one nonzero, empty rows
    ((80, 70, 66), (4, 64, 29), 2500, None),
    ((90, 3000), (6, 31), 7000, None),
    ((300, 64), (1, 64), 1000, 32),
    ((20, 24, 18, 15), (7, 5, 6, 3), 4000, None),
    ((30, 20, 25, 22), (16, 8, 9, 10), 3000, 32),   # 720 to 1,280 columns: several blocks of tiles
    ((12, 10, 11, 9, 8), (5, 4, 3, 5, 2), 3000, None),
    ((6, 7, 5, 6, 5, 4, 4, 3), (3, 2, 2, 3, 2, 2, 1, 2), 2000, None),
]


def make(dims, ranks, nnz):
    rng = np.random.default_rng(zlib.crc32(repr((dims, ranks, nnz)).encode()))
    coords = np.stack([rng.integers(0, d, nnz) for d in dims]).astype(np.uint32)
    vals = rng.standard_normal(nnz).astype(np.float32)
    return coords, vals, [rng.standard_normal((d, r)) for d, r in zip(dims, ranks)]


def check(T, ctx, dims, ranks, coords, vals, U):
    cc, cv = oracle.coalesce(coords, vals.astype(np.float64))
    cv = cv.astype(np.float32).astype(np.float64)  # as the context holds them
    for n in range(len(dims)):
        Y = T.ttmc_mode(ctx, n).cpu().numpy().astype(np.float64)
        ref = oracle.ttmc(dims, ranks, cc, cv, n, U)
        mag = oracle.ttmc(dims, ranks, cc, np.abs(cv), n, [np.abs(u) for u in U])
        k = np.bincount(cc[n], minlength=dims[n]).astype(np.float64)[:, None]
        chunk = T.tucker_mode_info(ctx, n)["chunk"]
        depth = np.minimum(k, chunk) + 31 + k / chunk + 8
        err = np.abs(Y - ref)
        bound = (depth + len(dims)) * 2.0 ** -24 * mag
        assert (err <= bound).all(), (n, float((err / np.maximum(bound, 1e-300)).max()))
        again = T.ttmc_mode(ctx, n).cpu().numpy()
        np.testing.assert_array_equal(again.astype(np.float64), Y)


@pytest.mark.parametrize("dims,ranks,nnz,chunk", CASES, ids=["x".join(map(str, c[1])) for c in CASES])
def test_tiled_ttmc(dims, ranks, nnz, chunk, monkeypatch):
    T = lib()
    if chunk:
        monkeypatch.setenv("TUCKER_TTMC_CHUNK", str(chunk))
    coords, vals, U = make(dims, ranks, nnz)
    ctx = T.tucker_init(dims, torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        [torch.as_tensor(u).cuda() for u in U])
    check(T, ctx, dims, ranks, coords, vals, f32_round(U))


@pytest.mark.parametrize("dims,ranks", [((50, 40, 30), (10, 12, 7)), ((30, 20, 25, 22), (4, 5, 8, 8))])
def test_bf16_factors_of_other_ranks(dims, ranks):
    T = lib()
    coords, vals, U = make(dims, ranks, 3000)
    ctx = T.tucker_init(dims, torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        [torch.as_tensor(u).cuda() for u in U], bf16=True)
    Ub = [torch.as_tensor(u).to(torch.bfloat16).double().numpy() for u in U]
    check(T, ctx, dims, ranks, coords, vals, Ub)


@pytest.mark.parametrize("ranks", [(8, 8, 8), (16, 16, 16), (10, 4, 7)])
def test_adjoint_with_factors_at_any_address(ranks):
    """Factors that start 4 bytes past a 16-byte boundary: the same loss and gradients, bit for bit."""
    T = lib()
    dims = (60, 50, 40)
    coords, vals, U = make(dims, ranks, 4000)
    ctx = T.tucker_init(dims, torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        [torch.as_tensor(u).cuda() for u in U])
    Uf = [torch.as_tensor(u, dtype=torch.float32).cuda() for u in U]
    G = torch.randn(ranks, generator=torch.Generator().manual_seed(3)).cuda()
    odd = []
    for u in Uf:
        b = torch.zeros(u.numel() + 1, device="cuda")
        b[1:] = u.reshape(-1)
        odd.append(b[1:].reshape(u.shape))
        assert odd[-1].data_ptr() % 16 == 4
    L, dU, dG = T.tucker_loss_grad(ctx, Uf, G)
    L2, dU2, dG2 = T.tucker_loss_grad(ctx, odd, G)
    assert torch.equal(L, L2) and torch.equal(dG, dG2) and all(torch.equal(a, b) for a, b in zip(dU, dU2))


def test_heavy_duplicates_sum_as_one_after_another():
    """Groups of equal coordinates of every length around the warp's 32 and the tile's 512 and
    8,192 positions: the values of the context are the FP64 sums in input order, rounded once, both
    where those sums are exact in any order and where (exponents 100 apart) they are not."""
    T = lib()
    rng = np.random.default_rng(5)
    lens = [1, 2, 31, 32, 33, 34, 127, 128, 129, 500, 512, 513, 2500, 8192, 9001, 1, 3]
    for spread in (0, 50):
        idx = np.concatenate([np.full(k, i) for i, k in enumerate(lens)])
        rng.shuffle(idx)
        vals = (rng.standard_normal(idx.size) * 2.0 ** rng.integers(-spread, spread + 1, idx.size)).astype(np.float32)
        coords = np.stack([idx % 5, idx // 5]).astype(np.uint32)
        ctx = T.tucker_init((5, 5), torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), (1, 1),
                            [torch.ones((5, 1), dtype=torch.float64).cuda() for _ in range(2)])
        want = np.zeros(25)
        for i, v in zip(idx, vals.astype(np.float64)):
            want[i] += v  # one after another
        assert T.tucker_nnz(ctx) == len(lens)
        np.testing.assert_allclose(T.tucker_norm2(ctx), (want ** 2).sum(), rtol=1e-14)
        dense = np.zeros((5, 5))
        dense.reshape(-1)[:] = 0
        for i in range(len(lens)):
            dense[i % 5, i // 5] = np.float32(want[i])
        for j in range(5):  # one column at a time: its entries are the context's values themselves
            e = torch.zeros((5, 1), dtype=torch.float64)
            e[j] = 1.0
            T.tucker_set_factor(ctx, 1, e.cuda())
            np.testing.assert_array_equal(T.ttmc_mode(ctx, 0).cpu().numpy()[:, 0].astype(np.float64), dense[:, j])


@pytest.mark.parametrize("rows", [4095, 4097, 70_000])
def test_units_of_many_slices(rows):
    """More slices than one round of the unit scan (4,096), and than its one block takes."""
    T = lib()
    rng = np.random.default_rng(rows)
    k = rng.integers(1, 4, rows)
    k[[0, rows // 2, rows - 1]] = 700  # cut slices at the ends
    i0 = np.repeat(np.arange(rows), k)
    coords = np.stack([i0, rng.integers(0, 50, i0.size), rng.integers(0, 60, i0.size)]).astype(np.uint32)
    vals = rng.standard_normal(i0.size).astype(np.float32)
    dims, ranks = (rows, 50, 60), (2, 3, 5)
    U = [rng.standard_normal((d, r)) for d, r in zip(dims, ranks)]
    ctx = T.tucker_init(dims, torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        [torch.as_tensor(u).cuda() for u in U])
    check(T, ctx, dims, ranks, coords, vals, f32_round(U))


@pytest.mark.parametrize("ranks", [(8, 29, 29), (8, 31, 32), (7, 30, 64)])
def test_steps_of_sixteen(ranks):
    """Records of 64 floats and more are taken 16 at a time: slices that end on either side of a step,
    and rows of four and eight chunks, whose tiles are numbered in another order."""
    T = lib()
    dims = (8, 90, 80)
    rng = np.random.default_rng(zlib.crc32(repr(ranks).encode()))
    i = np.repeat(np.arange(8), [1, 15, 16, 17, 31, 0, 33, 300])
    jk = np.stack(np.unravel_index(rng.permutation(90 * 80)[:i.size], (90, 80)))
    coords = np.concatenate([i[None], jk]).astype(np.uint32)
    vals = rng.standard_normal(i.size).astype(np.float32)
    U = [rng.standard_normal((d, r)) for d, r in zip(dims, ranks)]
    ctx = T.tucker_init(dims, torch.as_tensor(coords.astype(np.int32)).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        [torch.as_tensor(u).cuda() for u in U])
    check(T, ctx, dims, ranks, coords, vals, f32_round(U))
