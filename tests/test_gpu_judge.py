"""The judge of the learned proposal: the judge windows it opens (positions of uncovered local maxima of the
coarse spectrum, in order, sixteen at most) against a NumPy restatement, at coarse grids around the 256
points its lanes load together, with plateaus, NaN and covered maxima; and the rows it sends back."""
import numpy as np
import pytest

from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return require_gpu()


def _windows(p, clo, cstep, flo, fstep, Lf, first, width, jwidth):
    out = []
    Lc = len(p)
    for k in range(Lc):
        left = p[k] >= p[min(1, Lc - 1)] if k == 0 else p[k] > p[k - 1]
        right = k == Lc - 1 or p[k] >= p[k + 1]
        if not (left and right):
            continue
        c = int(np.rint((clo + k * cstep - flo) / fstep))
        f = max(0, min(c - jwidth // 2, Lf - jwidth))
        if not any(a >= 0 and a <= f and f + jwidth <= a + width for a in first):
            out.append(f)
    return out


@pytest.mark.parametrize("Lc", [3, 31, 33, 255, 256, 257, 513, 1801])
def test_judge_windows(env, Lc):
    torch, doa = env
    batch, M, dmax, width, jwidth, Lf = 37, 4, 2, 401, 21, 3601
    rng = np.random.default_rng(Lc)
    Pc = rng.random((batch, Lc)).astype(np.float32)
    smooth = rng.random((batch, Lc)).astype(np.float32)
    for _ in range(min(40, Lc)):
        smooth[:, 1:-1] = (smooth[:, :-2] + smooth[:, 1:-1] + smooth[:, 2:]) / np.float32(3)
    Pc[1::2] = smooth[1::2]                       # few maxima: no overflow of the sixteen windows
    Pc[2] = np.round(Pc[2] * 4)                   # plateaus
    Pc[3] = 1.0                                   # flat: a maximum at both ends' rules
    Pc[4, ::5] = np.nan
    win = rng.integers(0, Lf - width, (batch, dmax)).astype(np.int32)
    win[5::3, 1] = -1
    flo, fstep, clo, cstep = -90.0, 180.0 / (Lf - 1), -90.0, 180.0 / (Lc - 1)
    B = rng.standard_normal((batch, M * (M + 1), 2))
    K = np.full(batch, M - 1, np.int32)
    d = np.full(batch, 1, np.int32)
    val = np.full((batch, dmax), 1e30, np.float32)   # selected peaks that no judge window reaches
    val[7] = 0.0                                      # reached by any
    count = np.full(batch, 1, np.int32)
    count[9] = 0                                      # fewer peaks than asked for
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    jf = torch.full((batch, 16), -7, dtype=torch.int32, device="cuda")
    S = torch.zeros(Lf, dtype=torch.int32, device="cuda")
    Pj = torch.zeros((batch, 16, jwidth), device="cuda")
    fb = torch.zeros(batch, dtype=torch.int32, device="cuda")
    doa.doa_proposal_judge(dev(B).view(-1), M, dev(K), dev(d), dev(Pc), doa.grid(clo, cstep, Lc), doa.grid(flo, fstep, Lf),
                           dev(win), width, dev(val), dev(count), jwidth, jf, S, Pj, fb)
    torch.cuda.synchronize()
    jf, fb = jf.cpu().numpy(), fb.cpu().numpy()
    for r in range(batch):
        want = _windows(Pc[r], clo, cstep, flo, fstep, Lf, win[r], width, jwidth)
        got = list(jf[r][jf[r] >= 0])
        assert got == want[:16], r
        assert np.all(jf[r][len(got):] == -1)
        back = len(want) > 16 or count[r] < d[r] or (val[r, 0] == 0.0 and len(want) > 0)
        assert bool(fb[r]) == back, r
