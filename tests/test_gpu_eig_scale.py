"""The FP64 Jacobi at the ends of the range of doubles: a power of two times R has the same eigenvectors bit for
bit and that power times the eigenvalues."""
import numpy as np
import pytest

import oracle
from paper_2007_14135_gb300 import synth
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def decompose(torch, doa, R, d):
    M = R.shape[0]
    ev = torch.empty(M, dtype=torch.float64, device="cuda")
    B = torch.zeros(M * M, dtype=torch.complex128, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    doa.doa_noise_subspace_prec(torch.from_numpy(R).cuda(), d, doa.MUSIC, doa.EIG_FP64, B, info, evals=ev)
    torch.cuda.synchronize()
    return ev.cpu().numpy(), B.cpu().numpy(), info.item()


@pytest.mark.parametrize("M", [2, 5, 8, 13, 16, 31, 33, 64])
@pytest.mark.parametrize("exponent", [-900, -520, -300, 300, 520, 900])
def test_power_of_two_times_r(M, exponent):
    torch, doa = require_gpu()
    d = max(1, M // 4)
    R = oracle.covariance(synth.custom(M, d, 4 * M + 50, None, 10.0, 1.0, seed=850 + M).X)
    ev, B, info = decompose(torch, doa, R, d)
    assert info > 0
    got = decompose(torch, doa, R * 2.0 ** exponent, d)
    assert got[2] == info
    np.testing.assert_array_equal(got[0], ev * 2.0 ** exponent)
    np.testing.assert_array_equal(got[1], B)


def test_zero_and_graded_matrices():
    """A zero matrix, and a diagonal that spans 2^-700 .. 2^700."""
    torch, doa = require_gpu()
    ev, _, info = decompose(torch, doa, np.zeros((6, 6), complex), 2)
    assert info > 0 and not ev.any()
    w = 2.0 ** np.array([700.0, 10.0, -5.0, -700.0])
    ev, _, info = decompose(torch, doa, np.diag(w).astype(complex), 1)
    assert info > 0
    np.testing.assert_array_equal(ev, w)
