"""FP64 Grams and TTMs from the size where they run on exact integer digit
products on the tensor cores: against extended-precision sums, at the edges of
the tiles (128 x 64), of the 16-k stages and 128-k windows, in column and row
views, aligned or not, FP32 or FP64 input, and for operands outside the digit
range (NaN, Inf, rows of tiny magnitude), which take the FP64 pipe.

Bound per entry (u = 2^-53): every value is a 55-bit fixed-point number of its
row, off by at most 2^-55 of the row's largest magnitude; products below 2^-60
of the rows' maxima are left out; at most 152 partial sums are rounded to FP64
and added."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    """Digits for TTMs of every size (small ones are faster on the FP64 pipe)."""
    from paper_1901_06043_gb300 import tucker
    c = tucker.Context()
    c.set_option(tucker.OPT_FP64_KERNEL, tucker.FP64_KERNEL["digits"])
    yield c
    c.close()


def unfold(x, dims, mode):
    return np.moveaxis(np.reshape(x, dims, order="F"), mode, 0).reshape(dims[mode], -1)


def make(dims, mode, dtype, seed, spread):
    """Rows of very different size (one of zeros), entries over 12 decades
    when spread."""
    rng = np.random.default_rng(seed)
    I = dims[mode]
    shape = [1] * len(dims)
    shape[mode] = I
    x = rng.standard_normal(dims)
    if spread:
        x *= 10.0 ** rng.uniform(-12, 0, dims)
    x *= (10.0 ** rng.uniform(-6, 6, I)).reshape(shape)
    np.moveaxis(x, mode, 0)[I // 2] = 0.0
    # a value whose top digit is as large as it gets
    np.moveaxis(x, mode, 0)[0].flat[0] = np.nextafter(64.0 * 10 ** 6, 0)
    return np.reshape(x, -1, order="F").astype(dtype)


def dev(x, shift):
    """x on the device, its first element `shift` elements past an aligned address."""
    import torch
    t = torch.empty(x.size + shift, dtype=torch.float64 if x.dtype == np.float64 else torch.float32,
                    device="cuda")
    t[shift:] = torch.from_numpy(x).cuda()
    return t[shift:]


GRAMS = [  # dims, mode, shift
    ((64, 5000), 0, 0), ((64, 5000), 0, 1), ((65, 4801), 0, 0), ((127, 1601), 0, 0),
    ((128, 1300), 0, 1), ((129, 1217), 0, 0), ((192, 16, 37), 0, 0), ((200, 129, 7), 0, 0),
    ((500, 128), 0, 0), ((513, 100), 0, 0),
    ((2, 130, 700), 1, 0), ((3, 64, 1700), 1, 1), ((5, 7, 150, 31), 2, 0), ((33, 200, 19), 1, 0),
    ((1700, 129), 1, 0), ((16, 257, 33), 1, 0),
    # modes below 64, where K (I^2 - 565) reaches 6.5e7: one padded tile
    ((63, 22000), 0, 0), ((48, 45100), 0, 1), ((130, 60, 199), 1, 0), ((3, 50, 13000), 1, 1)]


@pytest.mark.parametrize("dtype,spread", [("f8", False), ("f8", True), ("f4", False)])
@pytest.mark.parametrize("dims,mode,shift", GRAMS)
def test_fp64_gram_on_digits(ctx, dims, mode, shift, dtype, spread):
    x = make(dims, mode, dtype, 1, spread)
    got = ctx.gram(dev(x, shift), dims, mode, prec="fp64").cpu().numpy()
    U = unfold(x, dims, mode).astype(np.longdouble)
    K = U.shape[1]
    want = U @ U.T
    A = np.abs(U).astype(np.float64)
    mx, one, two = A.max(1), A.sum(1), np.sqrt((A * A).sum(1))
    bound = (2.0 ** -55 * (np.outer(mx, one) + np.outer(one, mx)) + K * 2.0 ** -60 * np.outer(mx, mx)
             + 154 * 2.0 ** -53 * np.outer(two, two))
    assert np.array_equal(got, got.T)
    assert (np.abs(got - want) <= bound).all()


TTMS = [  # dims, mode, K, shift
    ((64, 129), 0, 1, 0), ((65, 128), 0, 64, 1), ((200, 401), 0, 65, 0), ((128, 127), 0, 28, 0),
    ((145, 300), 0, 33, 0), ((33, 64, 12), 1, 64, 0), ((4, 130, 70), 1, 129, 0),
    ((8, 130, 70), 1, 20, 1), ((7, 100, 31), 1, 17, 0), ((130, 16, 200), 1, 65, 0),
    ((3, 17, 33, 70), 2, 200, 0), ((40, 48, 64), 2, 54, 0), ((26, 9000), 0, 100, 0)]


@pytest.mark.parametrize("dtype", ["f8", "f4"])
@pytest.mark.parametrize("dims,mode,K,shift", TTMS)
def test_fp64_ttm_on_digits(ctx, dims, mode, K, shift, dtype):
    import torch
    from paper_1901_06043_gb300 import tucker
    x = make(dims, mode, dtype, 2, dtype == "f8")
    rng = np.random.default_rng(3)
    A = rng.standard_normal((K, dims[mode]))
    U = unfold(x, dims, mode)
    want = A.astype(np.longdouble) @ U.astype(np.longdouble)
    a, u = np.abs(A), np.abs(U).astype(np.float64)
    bound = (2.0 ** -55 * (np.outer(a.max(1), u.sum(0)) + np.outer(a.sum(1), u.max(0)))
             + dims[mode] * 2.0 ** -60 * np.outer(a.max(1), u.max(0)) + 2.0 ** -52 * np.abs(want))
    zd = list(dims)
    zd[mode] = K
    for arow in (True, False):
        At = torch.from_numpy(A).cuda() if arow else torch.from_numpy(A.T.copy()).cuda().t()
        z = ctx.ttm(dev(x, shift), dims, mode, At, prec="fp64", out_dtype=tucker.F64).cpu().numpy()
        assert (np.abs(unfold(z, zd, mode) - want) <= bound).all()
        z4 = ctx.ttm(dev(x, shift), dims, mode, At, prec="fp64", out_dtype=tucker.F32).cpu().numpy()
        assert np.array_equal(z4, z.astype(np.float32))


@pytest.mark.parametrize("what", ["nan", "inf", "tiny", "denormal"])
def test_fp64_digits_out_of_range_take_the_fp64_pipe(ctx, what):
    """The same special values as plain FP64 sums, and full relative precision
    of rows whose largest magnitude is below the digits' range."""
    import torch
    rng = np.random.default_rng(4)
    dims, K = (130, 1400), 30
    X = rng.standard_normal(dims)
    if what == "nan":
        X[5, 7] = np.nan
    elif what == "inf":
        X[5, 7], X[9, 3] = np.inf, -np.inf
    elif what == "tiny":
        X[5] *= 1e-295
    else:
        X[5] = 0.0
        X[5, 11] = 5e-324
    A = rng.standard_normal((K, dims[0]))
    x = torch.from_numpy(np.reshape(X, -1, order="F").copy()).cuda()
    with np.errstate(all="ignore"):
        for got, want, scale in (
                (ctx.gram(x, dims, 0, prec="fp64").cpu().numpy(), X @ X.T, np.abs(X) @ np.abs(X).T),
                (ctx.ttm(x, dims, 0, torch.from_numpy(A).cuda(), prec="fp64").cpu().numpy()
                 .reshape((K, -1), order="F"), A @ X, np.abs(A) @ np.abs(X))):
            fin = np.isfinite(want)
            assert np.array_equal(np.isnan(got), np.isnan(want))
            assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
            assert (np.abs(got - want)[fin] <= 1400 * 2.0 ** -52 * scale[fin] + 1e-322).all()


def graded(n, m, seed):
    """Fibres whose entries fall over 40 binary digits, in an order of their own each."""
    rng = np.random.default_rng(seed)
    e = np.linspace(0, -40, n)
    return np.stack([np.ldexp(rng.uniform(1, 2, n), e[rng.permutation(n)].astype(int))
                     * rng.choice([-1.0, 1.0], n) for _ in range(m)], 1)


@pytest.mark.parametrize("arow", [True, False])
@pytest.mark.parametrize("what", ["identity", "selection", "difference"])
def test_operators_with_zeros_keep_small_entries(ctx, what, arow):
    """An operator that leaves values of a fibre out: the entries it takes are as exact as
    in FP64 sums however large the others are."""
    import torch
    n, m = 96, 600
    X = graded(n, m, 5)
    A = np.eye(n)
    if what == "selection":
        A = A[3::7] * 0.75
    elif what == "difference":
        A = (np.eye(n) - np.eye(n, k=1))[:-1]
    x = torch.from_numpy(np.reshape(X, -1, order="F").copy()).cuda()
    At = torch.from_numpy(A).cuda() if arow else torch.from_numpy(A.T.copy()).cuda().t()
    z = ctx.ttm(x, (n, m), 0, At, prec="fp64").cpu().numpy().reshape((len(A), m), order="F")
    want = A.astype(np.longdouble) @ X.astype(np.longdouble)
    # (two terms at most: one product rounding each and one of the sum)
    assert (np.abs(z - want) <= 2.0 ** -52 * (np.abs(A) @ np.abs(X))).all()


@pytest.mark.parametrize("dims,mode", [((96, 4000), 0), ((5, 96, 900), 1), ((40, 70000), 0)])
def test_the_fp64_pipe_on_request(dims, mode):
    """TUCKER_OPT_FP64_KERNEL: entries to the rounding of FP64 sums, n 2^-53 sum |x| |y|,
    where rows differ by 40 binary digits within themselves."""
    import torch
    from paper_1901_06043_gb300 import tucker
    c = tucker.Context()
    c.set_option(tucker.OPT_FP64_KERNEL, tucker.FP64_KERNEL["pipe"])
    I, K = dims[mode], int(np.prod(dims)) // dims[mode]
    U = graded(K, I, 6).T                       # rows graded along the columns
    full = np.moveaxis(U.reshape([I] + [d for k, d in enumerate(dims) if k != mode], order="F"), 0, mode)
    x = torch.from_numpy(np.reshape(full, -1, order="F").copy()).cuda()
    U = unfold(np.reshape(full, -1, order="F"), dims, mode)
    S = c.gram(x, dims, mode, prec="fp64").cpu().numpy()
    L = U.astype(np.longdouble)
    assert (np.abs(S - L @ L.T) <= K * 2.0 ** -53 * (np.abs(U) @ np.abs(U).T)).all()
    A = graded(I, 33, 7).T
    z = c.ttm(x, dims, mode, torch.from_numpy(A).cuda(), prec="fp64").cpu().numpy()
    zd = list(dims)
    zd[mode] = 33
    assert (np.abs(unfold(z, zd, mode) - A.astype(np.longdouble) @ L)
            <= (I + 1) * 2.0 ** -53 * (np.abs(A) @ np.abs(U))).all()
    with pytest.raises(tucker.TuckerError):
        c.set_option(tucker.OPT_FP64_KERNEL, 3)
    c.close()


@pytest.mark.parametrize("dims,mode,K,digits", [((64, 1500), 0, 4, False), ((96, 6000), 0, 4, False),
                                                ((10, 64, 150), 1, 16, False), ((16, 24000), 0, 64, False),
                                                ((64, 1500), 0, 28, False), ((10, 64, 150), 1, 28, False),
                                                ((64, 24000), 0, 28, True), ((300, 64, 80), 1, 28, True),
                                                ((200, 24000), 0, 4, True), ((16, 100000), 0, 28, True)])
def test_ttm_takes_the_faster_kernel(dims, mode, K, digits):
    """The FP64 pipe's kernel (one launch) or the digits (three), by the work of both."""
    import torch
    from paper_1901_06043_gb300 import tucker
    ctx = tucker.Context()
    x = torch.randn(int(np.prod(dims)), device="cuda", dtype=torch.float64)
    A = torch.randn(K, dims[mode], device="cuda", dtype=torch.float64)
    n0 = tucker.kernel_launches()
    z = ctx.ttm(x, dims, mode, A, prec="fp64")
    assert tucker.kernel_launches() - n0 == (3 if digits else 1)
    X = x.cpu().numpy().reshape(dims, order="F")
    want = np.tensordot(A.cpu().numpy(), X, (1, mode))
    got = np.moveaxis(z.cpu().numpy().reshape([K if k == mode else d for k, d in enumerate(dims)],
                                              order="F"), mode, 0)
    assert np.abs(got - want).max() <= 1e-14 * dims[mode] * np.abs(want).max()
    ctx.close()


def test_batched_tensors_with_tiny_slices(ctx):
    """A batch does not wait for the verdict on each step; a slice below the digits' range
    (here 1e-295 of the others) is as good as zero there, as it is in the norm."""
    from paper_1901_06043_gb300 import synth
    import torch
    dims = (70, 80, 90)
    x, _ = synth.tucker_numpy(dims, (9, 8, 7), decay=0.2, eta=1e-6, seed=3)
    x = np.asarray(x, dtype=np.float64).reshape(dims, order="F")
    x[5] *= 1e-295
    x[:, 7] *= 1e-295
    xs = torch.from_numpy(x.reshape(-1, order="F").copy()).cuda()
    one = ctx.sthosvd(xs, dims, eps=1e-4, prec="fp64")
    many = ctx.sthosvd_batched([xs, xs], [dims, dims], eps=1e-4, prec="fp64")
    whole = one.reconstruct().cpu().numpy()
    for r in many:
        assert r.ranks == one.ranks
        # both are within eps of x; between them, the last kept vectors turn by rounding
        # over their gap: 1e-9 as for single steps of this size
        assert np.linalg.norm(r.reconstruct().cpu().numpy() - whole) <= 1e-9 * np.linalg.norm(whole)
