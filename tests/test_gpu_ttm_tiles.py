"""The TTM on the FP32 and FP64 pipes at the edges of its tiles: outputs around the tile
widths (8, 16, 24, 32 and several tiles), products below and above a block's m and
above the size from which a thread takes several, contraction lengths around a
stage of 32, column views (L = 1) and row views, unaligned inputs.

Bound per entry: the sum of I products in order, I u sum |a||y| with u = 2^-24 (FP32:
and both operands rounded once, 2 u) or 2^-53, and one rounding of an FP32 result.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1901_06043_gb300 import tucker
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    c = tucker.Context()
    yield c
    c.close()


VIEWS = [  # dims, mode
    ((1, 1), 0), ((5, 127), 0), ((31, 129), 0), ((32, 40), 0), ((33, 700), 0), ((47, 90000), 0),
    ((3, 5), 1), ((128, 31), 1), ((7, 33, 19), 1), ((129, 40, 1), 1), ((11, 13, 32), 2),
    ((301, 9, 120), 1), ((400, 33, 300), 1)]


@pytest.mark.parametrize("dims,mode", VIEWS)
@pytest.mark.parametrize("K", [1, 8, 9, 17, 24, 25, 32, 33, 70])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_ttm_tiles(ctx, dims, mode, K, prec):
    from paper_1901_06043_gb300 import tucker
    rng = np.random.default_rng(K + dims[0])
    x = rng.standard_normal(int(np.prod(dims)))
    A = rng.standard_normal((K, dims[mode]))
    U = np.moveaxis(x.reshape(dims, order="F"), mode, 0).reshape(dims[mode], -1)
    scale = np.abs(A) @ np.abs(U)
    want = A @ U
    zd = list(dims)
    zd[mode] = K
    buf = torch.empty(x.size + 1, device="cuda", dtype=torch.float32 if prec == "fp32" else torch.float64)
    t = buf[1:]
    t.copy_(torch.from_numpy(x))
    I = dims[mode]
    for arow in (True, False):
        At = torch.from_numpy(A).cuda() if arow else torch.from_numpy(A.T.copy()).cuda().t()
        for out in (tucker.F32, tucker.F64):
            z = ctx.ttm(t, dims, mode, At, prec=prec, out_dtype=out).double().cpu().numpy()
            z = np.moveaxis(z.reshape(zd, order="F"), mode, 0).reshape(K, -1)
            u = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
            bound = (I + 3) * u * scale + (2.0 ** -24 * np.abs(want) if out == tucker.F32 else 0.0)
            assert (np.abs(z - want) <= bound).all()


@pytest.mark.parametrize("dims", [(51, 12, 40), (64, 16, 3), (65, 16, 7), (128, 17, 9), (2999, 7, 5), (31, 16, 33),
                                  (51, 33, 40), (65, 48, 7), (65, 49, 7), (64, 40, 9)])
@pytest.mark.parametrize("K", [32, 33, 63, 64, 65, 130])
def test_row_views_of_few_rows(ctx, dims, K):
    """FP32 row views around the lines between the 64 x 64 tiles (at most 16 rows, or 33 to 48
    without 16-byte loads, more than 32 outputs, half of the tiles' entries used) and the
    narrower ones; bound as above."""
    rng = np.random.default_rng(K + dims[0])
    x = rng.standard_normal(dims).astype(np.float32)
    A = rng.standard_normal((K, dims[1]))
    want = np.einsum("ki,lir->lkr", A, x.astype(np.float64))
    scale = np.einsum("ki,lir->lkr", np.abs(A), np.abs(x).astype(np.float64))
    xt = torch.from_numpy(x.reshape(-1, order="F").copy()).cuda()
    for At in (torch.from_numpy(A).cuda(), torch.from_numpy(A.T.copy()).cuda().t()):
        z = ctx.ttm(xt, dims, 1, At, prec="fp32").double().cpu().numpy()
        z = z.reshape((dims[0], K, dims[2]), order="F")
        assert (np.abs(z - want) <= (dims[1] + 3) * 2.0 ** -24 * scale).all()


@pytest.mark.parametrize("dims,mode", [((3, 4), 0), ((2, 3, 2), 1)])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_more_output_tiles_than_a_grid_dimension(ctx, dims, mode, prec):
    """2.2 million outputs: 68,751 tiles of 32."""
    K = 2200001
    gen = torch.Generator("cuda").manual_seed(3)
    dt = torch.float32 if prec == "fp32" else torch.float64
    x = torch.randn(12, device="cuda", generator=gen, dtype=dt)
    A = torch.randn(K, 3, device="cuda", generator=gen, dtype=torch.float64)
    z = ctx.ttm(x, dims, mode, A, prec=prec).double()
    U = x.double().reshape(tuple(reversed(dims)))
    if mode == 0:
        got, want, scale = z.reshape(4, K), U @ A.T, U.abs() @ A.abs().T
    else:
        got, want, scale = z.reshape(2, K, 2), A @ U, A.abs() @ U.abs()
    u = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
    assert bool(((got - want).abs() <= 6 * u * scale).all())


@pytest.mark.parametrize("dims,mode,K", [((40, 128), 0, 17), ((500, 384), 0, 100), ((16, 33, 7), 1, 300),
                                         ((132, 54, 3), 1, 513), ((128, 5, 2), 1, 1)])
@pytest.mark.parametrize("scale", [1e-25, 1.0, 1e12])
@pytest.mark.parametrize("arow", [True, False])
def test_mixed_operator_images(ctx, dims, mode, K, scale, arow):
    """The tensor-core TTM's operator images at any scale of the operator, rows of very
    different size, and a NaN that leaves the other outputs alone.  Both operands are
    rounded to 22 bits of their largest value and three of the four products kept:
    1e-5 of sum |a|max |y| covers I <= 500 products and the FP32 accumulation."""
    from paper_1901_06043_gb300 import tucker
    rng = np.random.default_rng(K)
    x = rng.standard_normal(int(np.prod(dims))).astype(np.float32)
    A = rng.standard_normal((K, dims[mode])) * scale * 10.0 ** rng.uniform(-8, 0, (K, 1))
    U = np.moveaxis(x.astype(np.float64).reshape(dims, order="F"), mode, 0).reshape(dims[mode], -1)
    bound = 1e-5 * np.abs(A).max() * np.abs(U).sum(0)
    zd = list(dims)
    zd[mode] = K
    for nan in (False, True):
        B = A.copy()
        if nan:
            B[K // 2, 3] = np.nan
        want = B @ U
        At = torch.from_numpy(B).cuda() if arow else torch.from_numpy(B.T.copy()).cuda().t()
        z = ctx.ttm(torch.from_numpy(x).cuda(), dims, mode, At, prec="mixed", out_dtype=tucker.F32)
        z = z.double().cpu().numpy().reshape(zd, order="F")
        z = np.moveaxis(z, mode, 0).reshape(K, -1)
        fin = np.isfinite(want)
        assert np.array_equal(np.isfinite(z), fin)
        assert (np.abs(z - want)[fin] <= np.broadcast_to(bound, want.shape)[fin]).all()
