"""Rows of slices that are cut over several work units: the pieces' partial rows are added by one warp for
each 128, 64 or 32 columns of a row up to 16 pieces, and by a block for 32 columns for more.  Numbers of pieces
on both sides of 8 (one round of loads) and 16, widths that are and are not multiples of 2, 32 and 64; and enough
slices for 128 columns a warp.

Bar: the componentwise bound of test_gpu_ttmc_tile.py, (depth + order) 2^-24 of sum |x| prod |u|; a row of L
nonzeros in pieces of 32 is a sum of at most 32 + L / 32 + 8 terms deep."""
import numpy as np
import pytest

from tests.gpu_util import lib, torch

pytestmark = pytest.mark.gpu

LENGTHS = [33, 64, 65, 256, 257, 288, 512, 513, 1056, 9000, 1, 32, 5]  # nonzeros of the slices of mode 1


@pytest.mark.parametrize("ranks", [(3, 16, 16), (3, 8, 8), (2, 32, 32), (3, 5, 3), (3, 2, 10), (2, 33, 33), (4, 6, 22)],
                         ids=lambda r: "x".join(map(str, r)))
def test_pieces(ranks, monkeypatch):
    T = lib()
    monkeypatch.setenv("TUCKER_TTMC_CHUNK", "32")
    rng = np.random.default_rng(sum(ranks))
    dims = (len(LENGTHS) + 2, 150, 140)
    rows, cells = [], []
    for i, n in enumerate(LENGTHS):
        rows += [i + 1] * n  # (rows 0 and the last are empty)
        cells += list(rng.choice(dims[1] * dims[2], size=n, replace=False))
    cells = np.array(cells)
    coords = np.stack([rows, cells // dims[2], cells % dims[2]]).astype(np.int32)
    vals = rng.standard_normal(len(rows)).astype(np.float32)
    U = [rng.standard_normal((d, r)).astype(np.float32) for d, r in zip(dims, ranks)]
    ctx = T.tucker_init(dims, torch.as_tensor(coords).cuda(), torch.as_tensor(vals).cuda(), ranks,
                        [torch.as_tensor(u.astype(np.float64)).cuda() for u in U])
    assert T.tucker_mode_info(ctx, 0)["long_slices"] == sum(n > 32 for n in LENGTHS)
    Y = T.ttmc_mode(ctx, 0)
    P = ctx.P(0)
    Y = Y.double().cpu().numpy()
    K = (U[1].astype(np.float64)[coords[1]][:, :, None] * U[2].astype(np.float64)[coords[2]][:, None, :]).reshape(-1, P)
    K *= vals.astype(np.float64)[:, None]
    for i, n in enumerate(LENGTHS):
        k = K[coords[0] == i + 1]
        bound = (32 + n / 32 + 8 + 3) * 2.0**-24 * np.abs(k).sum(0)
        assert (np.abs(Y[i + 1] - k.sum(0)) <= bound).all(), n
    assert not Y[0].any() and not Y[-1].any()
    T.tucker_free(ctx)


@pytest.mark.parametrize("ranks", [(2, 16, 16), (2, 12, 11)], ids=lambda r: "x".join(map(str, r)))
def test_many_slices(ranks, monkeypatch):
    """3,000 slices of 33 to 600 nonzeros, by 128 columns a warp, against the same slices in pieces of 1,024
    (none cut): sums of at most 600 products in other orders, each within 600 2^-24 of sum |x| prod |u|."""
    T = lib()
    rng = np.random.default_rng(7)
    dims, lengths = (3000, 90, 80), rng.integers(33, 600, 3000)
    rows = np.repeat(np.arange(3000), lengths)
    cells = np.concatenate([rng.choice(90 * 80, n, replace=False) for n in lengths])
    coords = torch.as_tensor(np.stack([rows, cells // 80, cells % 80]).astype(np.int32)).cuda()
    vals = torch.as_tensor(rng.standard_normal(len(rows)).astype(np.float32)).cuda()
    U = [torch.as_tensor(rng.standard_normal((d, r)).astype(np.float32).astype(np.float64)).cuda() for d, r in zip(dims, ranks)]
    monkeypatch.setenv("TUCKER_TTMC_FIBERS", "0")
    out = []
    for chunk, x, u in ((32, vals, U), (1024, vals, U), (1024, vals.abs(), [a.abs() for a in U])):
        monkeypatch.setenv("TUCKER_TTMC_CHUNK", str(chunk))
        ctx = T.tucker_init(dims, coords, x, ranks, u)
        assert T.tucker_mode_info(ctx, 0)["long_slices"] == (3000 if chunk == 32 else 0)
        out.append(T.ttmc_mode(ctx, 0).double())
        T.tucker_free(ctx)
    assert ((out[0] - out[1]).abs() <= 2 * 600 * 2.0**-24 * out[2] * 1.001).all()


def test_norms_of_cut_slices(monkeypatch):
    """The squares of the finished entries (ttmc_mode_norms): each exact, summed in double-float."""
    T = lib()
    monkeypatch.setenv("TUCKER_TTMC_CHUNK", "32")
    rng = np.random.default_rng(1)
    n = 40_000
    coords = np.stack([np.minimum(rng.geometric(0.02, n), 399), rng.integers(0, 150, n), rng.integers(0, 140, n)])
    ctx = T.tucker_init((400, 150, 140), torch.as_tensor(coords.astype(np.int32)).cuda(),
                        torch.as_tensor(rng.standard_normal(n).astype(np.float32)).cuda(), (8, 16, 16), seed=2)
    info = T.tucker_mode_info(ctx, 0)
    assert 0 < info["long_slices"] < info["slices"]
    Y, sq = T.ttmc_mode_norms(ctx, 0)
    assert torch.equal(Y, T.ttmc_mode(ctx, 0))
    np.testing.assert_allclose(sq.cpu().numpy(), (Y.double() ** 2).sum(0).cpu().numpy(), rtol=1e-12)
    T.tucker_free(ctx)
