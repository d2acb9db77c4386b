"""Single FP32 covariances split over clusters: the block ranges and snapshot ranges at their edges."""
import numpy as np
import pytest

import oracle
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,pad", [(2, 1, 0), (3, 127, 0), (4, 128, 3), (5, 129, 0), (8, 1024, 0), (16, 255, 1), (17, 1000, 0),
                                     (33, 4099, 5), (63, 2048, 0), (64, 16384, 0), (64, 130, 0)])
def test_single_covariance_matches_oracle(M, N, pad):
    """Compensated sums: 1e-12 of max |R| against the FP64 oracle (2^-44 relative to the sums of |terms|),
    Hermitian exactly."""
    torch, doa = require_gpu()
    rng = np.random.default_rng(1000 * M + N)
    X = (rng.standard_normal((M, N + pad)) + 1j * rng.standard_normal((M, N + pad))).astype(np.complex64)
    Xd = torch.from_numpy(X).cuda()[:, :N]
    R = torch.full((M, M), float("nan"), dtype=torch.complex128, device="cuda")
    doa.doa_covariance(Xd, R64=R)
    torch.cuda.synchronize()
    got, want = R.cpu().numpy(), oracle.covariance(np.ascontiguousarray(X[:, :N]))
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    assert np.array_equal(got, got.conj().T)
