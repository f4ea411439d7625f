"""The truncated eigensolve's Cholesky QR at the edges of its blocks (one CTA
up to 64 vectors, then blocks of 32), with well separated eigenvalues (one
pass) and with clusters (two passes): orthonormal vectors and small residuals."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1901_06043_gb300 import tucker
    c = tucker.Context()
    yield c
    c.close()


@pytest.mark.parametrize("clustered", [False, True])
@pytest.mark.parametrize("n,R", [(5, 1), (33, 31), (40, 32), (70, 33), (100, 63), (100, 64),
                                 (100, 65), (200, 96), (200, 97), (300, 161), (257, 257)])
def test_vectors_are_orthonormal_eigenvectors(ctx, n, R, clustered):
    import torch
    rng = np.random.default_rng(n + R)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.sort(10.0 ** np.linspace(0, -6, n))[::-1]
    if clustered:                       # runs of three within 1e-9 of each other
        lam = lam[(np.arange(n) // 3) * 3] * (1 + 1e-9 * (np.arange(n) % 3))
        lam = np.sort(lam)[::-1]
    S = (Q * lam) @ Q.T
    S = (S + S.T) / 2
    w, U, k, _ = ctx.eig_trunc(torch.from_numpy(S).cuda(), R=R)
    w, U = w.cpu().numpy(), U.cpu().numpy()
    assert k == R and np.abs(w - lam).max() <= 1e-13 * n
    assert np.abs(U.T @ U - np.eye(R)).max() <= 1e-13 * n
    assert np.abs(S @ U - U * w[:R]).max() <= 1e-13 * n


def test_second_pass_is_launched_only_where_needed(ctx):
    """Above 64 vectors the second pass (its Gram and the factor's blocks) is not launched
    for well separated eigenvalues."""
    import torch
    from paper_1901_06043_gb300 import tucker
    n, R = 200, 97
    rng = np.random.default_rng(0)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    counts = []
    for lam in (np.linspace(2, 1, n), np.repeat(np.linspace(2, 1, n // 4), 4)):
        S = (Q * lam) @ Q.T
        St = torch.from_numpy((S + S.T) / 2).cuda()
        before = tucker.kernel_launches()
        _, U, _, _ = ctx.eig_trunc(St, R=R)
        counts.append(tucker.kernel_launches() - before)
        U = U.cpu().numpy()
        assert np.abs(U.T @ U - np.eye(R)).max() <= 1e-13 * n
    # two launches of the Gram, 3 * 3 + 1 of the four blocks' factor, one of the product
    assert counts[0] + 12 <= counts[1]


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 1023, 1024, 1025, 2500])
def test_rank_cut_sums_in_order(ctx, n):
    """Bitwise the sequential sum from the smallest value up, also across the
    kernel's chunks of 1024."""
    import torch
    rng = np.random.default_rng(n)
    w = np.sort(10.0 ** rng.uniform(-12, 0, n))[::-1] * np.where(np.arange(n) > n // 2, -1.0, 1.0)
    tail = np.zeros(n + 1)
    for i in range(n - 1, -1, -1):
        tail[i] = tail[i + 1] + w[i]
    for thr in (0.0, abs(tail[n // 3]), 1e-6, 10.0 * n):
        R, d = ctx.rank_cut(torch.from_numpy(w).cuda(), thr)
        want = next(r for r in range(1, n + 1) if tail[r] <= thr)
        assert (R, d) == (want, tail[want])


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 16, 17, 31, 47, 64, 129, 153, 304, 305, 610,
                               640, 641, 1000])
@pytest.mark.parametrize("kind", ["dense", "diagonal", "split", "tiny", "huge"])
def test_eigenvalues_and_vectors_over_sizes(ctx, n, kind):
    """The widths of the multisection that one matrix takes (four warps per eigenvalue to
    16 lanes; narrower ones in test_gpu_batch_regimes.py), the two-ended inverse
    iteration at odd and even sizes, both exchanges of the reduction (words up to 640
    rows, a barrier above), exact zeros on T's off-diagonal and matrices near the ends of
    the exponent range."""
    import torch
    rng = np.random.default_rng(n)
    S = rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-3, 0, n)
    S = S @ S.T
    if kind == "diagonal":
        S = np.diag(10.0 ** rng.uniform(-9, 0, n))
    elif kind == "split":
        h = n // 2
        S[h:, :h] = S[:h, h:] = 0.0
    scale = {"tiny": 2.0 ** -480, "huge": 2.0 ** 480}.get(kind, 1.0)
    lam, _ = np.linalg.eigh(S)
    lam = lam[::-1]
    R = max(1, n // 3)
    w, U, k, _ = ctx.eig_trunc(torch.from_numpy(S * scale).cuda(), R=R)
    w, U = w.cpu().numpy() / scale, U.cpu().numpy()
    top = abs(lam).max()
    assert np.abs(w - lam).max() <= 1e-14 * n * top + 1e-15 * top
    assert np.abs(U.T @ U - np.eye(R)).max() <= 1e-13 * n
    assert np.abs(S @ U - U * w[:R]).max() <= 1e-13 * n * top
