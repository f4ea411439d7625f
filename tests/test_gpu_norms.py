"""The passes that read a tensor for its norm and its rows' largest values, at the
edges of their splits: odd and unaligned lengths, columns shorter and longer than a
block, one column more than the loads in flight.

Tolerances: an FP64 sum of n squares in any order is within n eps of its value,
and n eps <= 4e-10 here is far above what occurs, so 1e-13 (a block's partial sums
hold a few hundred terms).  The MIXED Gram of small integers times one power of two
per row is exact when every row's scale is its largest value's, so it is compared
for equality.
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


@pytest.mark.parametrize("n", [1, 2, 3, 511, 4097, 1245185, 1245200 + 7])
@pytest.mark.parametrize("off", [0, 1])
def test_norm_of_fp64_data(ctx, n, off):
    from paper_1901_06043_gb300 import tucker
    x = torch.zeros(n + off, device="cuda", dtype=torch.float64)[off:]
    x.copy_(torch.from_numpy(np.random.default_rng(n).standard_normal(n)))
    want = float((x.cpu().numpy().astype(np.longdouble) ** 2).sum())
    assert abs(ctx.norm_sq(x) - want) <= 1e-13 * want
    for bad in (float("inf"), float("-inf"), float("nan")):
        for at in (0, n // 2, n - 1):
            keep = float(x[at])
            x[at] = bad
            with pytest.raises(tucker.TuckerError) as e:
                ctx.norm_sq(x)
            assert e.value.name == "NONFINITE"
            x[at] = keep


@pytest.mark.parametrize("I", [64, 65, 100, 128, 129, 256, 257, 260, 300, 512, 516, 1030, 2052])
@pytest.mark.parametrize("cols", [640, 3001])
def test_row_maxima_set_the_digits(ctx, I, cols):
    rng = np.random.default_rng(I + cols)
    x = rng.integers(-7, 8, (cols, I)).astype(np.float64)
    # each row's largest value once, in the first, the last or any other column
    at = np.where(np.arange(I) % 3 == 0, 0, np.where(np.arange(I) % 3 == 1, cols - 1,
                                                     rng.integers(0, cols, I)))
    x[at, np.arange(I)] = 63.0 * rng.choice((-1.0, 1.0), I)
    x *= 2.0 ** rng.integers(-20, 20, I)
    t = torch.from_numpy(x.reshape(-1)).to(device="cuda", dtype=torch.float32)
    got = ctx.gram(t, (I, cols), 0, prec="mixed").cpu().numpy().reshape(I, I)
    assert np.array_equal(got, x.T @ x)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_norms_of_a_batch(ctx, dt):
    """Tensors of very different sizes, odd lengths and unaligned starts; NaN in one of them."""
    from paper_1901_06043_gb300 import tucker
    shapes = [(5, 3), (129, 65, 33), (7, 11, 13), (64, 50, 40), (255,), (3, 3, 3, 3)]
    xs = []
    for k, d in enumerate(shapes):
        n = int(np.prod(d))
        x = torch.zeros(n + k % 2, device="cuda", dtype=dt)[k % 2:]
        x.copy_(torch.from_numpy(np.random.default_rng(k).standard_normal(n) * 10.0 ** (k - 3)))
        xs.append(x)
    for r, x in zip(ctx.sthosvd_batched(xs, shapes, eps=1e-3, prec="fp64"), xs):
        want = float((x.double().cpu().numpy().astype(np.longdouble) ** 2).sum())
        assert abs(r.norm_sq - want) <= 1e-13 * want
        r.close()
    xs[3][-1] = float("nan")
    with pytest.raises(tucker.TuckerError) as e:
        ctx.sthosvd_batched(xs, shapes, eps=1e-3, prec="fp64")
    assert e.value.name == "NONFINITE"
