"""The data SVD on a stream that has only some of the SMs (a green context): its CTAs wait for one another, so it
takes no more of them than can be resident there."""
import ctypes

import numpy as np
import pytest

import oracle
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu
SM = 1                      # CU_DEV_RESOURCE_TYPE_SM


class Resource(ctypes.Structure):
    """CUdevResource: type, padding, and the SM member of its union."""
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sms", ctypes.c_uint), ("rest", ctypes.c_ubyte * 44)]


def partition_stream(cu, sms):
    """A stream of a green context of `sms` SMs or a few more, and their number; None where there are none."""
    p = ctypes.c_void_p
    whole, part, rest, n = Resource(), Resource(), Resource(), ctypes.c_uint(1)
    desc, green, stream = p(), p(), p()
    cu.cuStreamGetCtx.restype = ctypes.c_int
    steps = (lambda: cu.cuDeviceGetDevResource(0, ctypes.byref(whole), SM),
             lambda: cu.cuDevSmResourceSplitByCount(ctypes.byref(part), ctypes.byref(n), ctypes.byref(whole), ctypes.byref(rest), 0, sms),
             lambda: cu.cuDevResourceGenerateDesc(ctypes.byref(desc), ctypes.byref(part), 1),
             lambda: cu.cuGreenCtxCreate(ctypes.byref(green), desc, 0, 1),
             lambda: cu.cuGreenCtxStreamCreate(ctypes.byref(stream), green, 1, 0))
    for step in steps:
        if step() != 0:
            return None
    return stream.value, part.sms


@pytest.mark.parametrize("M,N", [(8, 4096), (16, 8192)])
def test_svd_in_a_green_context(M, N):
    torch, doa = require_gpu()
    got = partition_stream(ctypes.CDLL("libcuda.so.1"), 16)
    if got is None:
        pytest.skip("no green contexts here")
    handle, sms = got
    assert 16 <= sms < torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(M)
    X = (rng.standard_normal((M, N)) + 1j * rng.standard_normal((M, N))).astype(np.complex64)
    Xd = torch.from_numpy(X).cuda()
    ev = torch.zeros(M, dtype=torch.float64, device="cuda")
    U = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(doa.svd_data_ws_bytes(M, N), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    stream = torch.cuda.ExternalStream(handle)
    doa.doa_svd_data(Xd, ev, U, info, ws=ws, stream=stream)
    stream.synchronize()
    assert info.item() > 0
    want, _, _ = oracle.svd_data(X)
    np.testing.assert_allclose(ev.cpu().numpy(), want, rtol=1e-12)
