"""The batched truncated eigensolve where its launches differ most: as many tensors as
SMs or more, so that every team is one CTA (rows in shared memory up to 123, else in
global memory; one lane per eigenvalue in the bisection), with small and large modes in
one launch; fewer tensors, with a team behind a barrier (above 640 rows) beside teams that
exchange words.  Ranks and eigenvalues against the same tensor by itself."""
import numpy as np
import pytest

from paper_1901_06043_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1901_06043_gb300 import tucker
    c = tucker.Context()
    yield c
    c.close()


def check(ctx, sizes, seed):
    """A batch of thin tensors n x 6 x 5; one tensor of every size again by itself.  Both
    eigenvalues are within rounding of the matrix, ~n 2^-53 of its norm, of the exact."""
    xs = [torch.from_numpy(synth.tucker_numpy((n, 6, 5), (min(n, 4), 3, 3), decay=0.2, eta=1e-6,
                                              seed=seed + k)[0]).cuda()
          for k, n in enumerate(sizes)]
    dims = [(n, 6, 5) for n in sizes]
    many = ctx.sthosvd_batched(xs, dims, eps=1e-4, prec="fp64")
    seen = set()
    for x, d, r in zip(xs, dims, many):
        assert r.eig_kernel == ["tridiag"] * 3
        if d[0] not in seen:
            seen.add(d[0])
            one = ctx.sthosvd(x, d, eps=1e-4, prec="fp64")
            assert one.ranks == r.ranks
            for n, a, b in zip(d, one.eigvals, r.eigvals):
                assert float((a - b).abs().max()) <= 1e-14 * n * float(a[0]) + 1e-15 * float(a[0])
            one.close()
        full = r.reconstruct()
        assert float((full - x).norm()) <= 1e-4 * float(x.norm())
        r.close()


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def test_teams_of_one_with_small_and_large_modes(ctx):
    """2350 rows need 113 KB of vectors, 123 rows 118 KB for the matrix: each fits an SM,
    their sum does not."""
    rest = [3, 100, 123, 124, 300]
    sizes = [2350, 123, 700] + [rest[k % 5] for k in range(sms() - 2)]
    check(ctx, sizes, 500)


def test_a_team_behind_a_barrier_beside_teams_with_words(ctx):
    """100 tensors: 1000 rows in a team of some 30 CTAs, 640 and 641 beside it, the small
    ones mostly in teams of one."""
    sizes = [1000, 640, 641, 124, 123] + [20 + k for k in range(95)]
    check(ctx, sizes, 900)


def test_large_ranks_in_a_batch(ctx):
    """More than 64 vectors (blocks of 32, the second pass chosen on the host) beside fewer;
    well separated and clustered eigenvalues in one batch."""
    rng = np.random.default_rng(11)
    xs, dims = [], []
    for n, clustered in ((150, False), (150, True), (90, True), (40, False)):
        d = (n, 180, 2)
        Q = np.linalg.qr(rng.standard_normal((n, n)))[0]
        P = np.linalg.qr(rng.standard_normal((360, n)))[0]
        s = np.linspace(2, 1, n)
        if clustered:
            s = s[(np.arange(n) // 5) * 5]
        xs.append(torch.from_numpy(np.reshape((Q * s) @ P.T, -1, order="F").copy()).cuda())
        dims.append(d)
    many = ctx.sthosvd_batched(xs, dims, eps=0.1, prec="fp64")
    for x, d, r in zip(xs, dims, many):
        U = r.factors[0].cpu().numpy()
        R = r.ranks[0]
        assert U.shape == (d[0], R) and (d[0] < 90 or R > 64)
        assert np.abs(U.T @ U - np.eye(R)).max() <= 1e-13 * d[0]
        assert float((r.reconstruct() - x).norm()) <= 0.1 * float(x.norm())
        r.close()
