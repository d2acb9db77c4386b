"""The digits of a single FP32-mode covariance: an entry of R is the same chain of compensated additions
wherever its blocks are computed. Noise eigenvectors follow R's last digits, so the comparisons are exact:
against the per-chunk form (where its chunks are the single call's snapshot ranges) and against the sums
written out in NumPy."""
import numpy as np
import pytest

from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu
f32 = np.float32


@pytest.fixture(scope="module")
def env():
    return require_gpu()


def snapshots(M, N, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((M, N)) + 1j * rng.standard_normal((M, N))).astype(np.complex64)


def two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def df_add(x, y):
    s, e = two_sum(x[0], y[0])
    e = e + (x[1] + y[1])
    h = s + e
    return h, e - (h - s)


def mac(acc, a, b):
    """hi + lo += a b; the product's error is exact in 64 bits."""
    p = a * b
    e = (a.astype(np.float64) * b - p).astype(f32)
    s, t = two_sum(acc[0], p)
    return s, acc[1] + (e + t)


def covariance_in_order(X):
    M, N = X.shape
    mb = -(-M // 4)
    groups = max(1, 256 // (mb * (mb + 1) // 2))
    nc = min(8, -(-N // 1024))
    per = -(-N // nc)
    i, j = np.triu_indices(M)
    total = np.zeros((2, len(i)))
    for rank in range(nc):
        x = X[:, rank * per:min(N, (rank + 1) * per)]
        z = np.zeros((groups, len(i)), f32)
        re, im = (z, z), (z, z)
        for t0 in range(0, x.shape[1], 64):
            tile = x[:, t0:t0 + 64]
            for s in range(0, tile.shape[1], groups):
                a, b = tile[i, s:s + groups].T, tile[j, s:s + groups].T
                n = a.shape[0]
                r, m = tuple(v[:n] for v in re), tuple(v[:n] for v in im)
                r = mac(mac(r, a.real, b.real), a.imag, b.imag)
                m = mac(mac(m, a.imag, b.real), -a.real, b.imag)
                re = tuple(np.concatenate([u, v[n:]]) for u, v in zip(r, re))
                im = tuple(np.concatenate([u, v[n:]]) for u, v in zip(m, im))
        for k, acc in enumerate((re, im)):
            s = (acc[0][0], acc[1][0])
            for g in range(1, groups):
                s = df_add(s, (acc[0][g], acc[1][g]))
            total[k] += s[0].astype(np.float64) + s[1]
    R = np.zeros((M, M), complex)
    R[i, j] = (total[0] + 1j * np.where(i == j, 0.0, total[1])) * (1.0 / N)
    return np.where(np.arange(M)[:, None] <= np.arange(M)[None], R, R.T.conj())


def single(env, X, ld=None):
    torch, doa = env
    M, N = X.shape
    Xd = torch.zeros((M, ld or N), dtype=torch.complex64, device="cuda")
    Xd[:, :N] = torch.from_numpy(X)
    R = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
    doa.doa_covariance(Xd[:, :N], R64=R)
    return Xd[:, :N], R


@pytest.mark.parametrize("M", [2, 4, 5, 8, 9, 12, 16, 17, 28, 33, 48, 61, 64])
@pytest.mark.parametrize("N", [1, 63, 65, 1000, 1024, 2048, 5120, 8192])
def test_single_equals_per_chunk_form(env, M, N):
    torch, doa = env
    X, R = single(env, snapshots(M, N, 7 * M + N), N + N % 3)
    want = torch.zeros_like(R)
    doa.doa_covariance_noalloc(X, R64=want)
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(R), torch.view_as_real(want))


@pytest.mark.parametrize("M,N", [(3, 1500), (7, 3001), (9, 1025), (16, 9001), (33, 1500), (64, 1030)])
def test_single_equals_sums_in_order(env, M, N):
    torch, doa = env
    X = snapshots(M, N, 11 * M + N)
    _, R = single(env, X)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(R.cpu().numpy(), covariance_in_order(X))
