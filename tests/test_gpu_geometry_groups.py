"""Shared-steering geometry scan: the problems that share a steering table scanned in groups, against
the same problems scanned one by one (spectra and peaks bit for bit), at ragged tiles, group sizes that
do not divide the problems, M below the padded size, and every readout subset's columns."""
import numpy as np
import pytest

from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return require_gpu()


# (M, La, Le, problems, mask, d)
CASES = [
    (8, 360, 90, 307, 0xF, 2),
    (8, 97, 333, 309, 0x2, 2),
    (5, 361, 89, 331, 0xF, 1),
    (8, 361, 89, 310, 0x9, 0),
    (16, 97, 13, 1001, 0xF, 3),
    (11, 361, 30, 150, 0x6, 4),
]


@pytest.mark.parametrize("M,La,Le,B,mask,d", CASES)
def test_groups_match_single_problems(env, M, La, Le, B, mask, d):
    torch, doa = env
    N, npts, na = 64, La * Le, bin(mask).count("1")
    rng = np.random.default_rng(1000 * M + B)
    t = 2.0 * np.pi * np.arange(M) / M
    pos = torch.from_numpy(np.stack([0.5 * np.cos(t), 0.5 * np.sin(t), 0.1 * rng.standard_normal(M)], axis=1)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(M * 7 + B)
    X = torch.randn(B, M, N, 2, generator=gen, device="cuda", dtype=torch.float32)
    X[:, 1:, :, 0] += 0.8 * X[:, :1, :, 0]         # some correlation: spectra with structure
    X = torch.view_as_complex(X)
    step = 360.0 / La
    out = []
    for group in (None, (1, 1, 1, 1)):
        P = torch.full((B, na * npts + 1), -1.0, device="cuda")
        dk = max(d, 1)
        idx = torch.full((B, na * dk), -1, dtype=torch.int32, device="cuda")
        val = torch.zeros((B, na * dk), device="cuda")
        cnt = torch.zeros((B, na), dtype=torch.int32, device="cuda")
        probs = [doa.make_problem(X[i], d, mask, doa.grid(0.0, step, La), P[i, :-1], idx[i] if d else None,
                                  val[i] if d else None, cnt[i], None,
                                  geom=doa.geometry(pos, 2.0, 0.9, Le, La % 2 == 0)) for i in range(B)]
        plan = doa.BatchPlan(probs, scan_group=group)
        groups = int(plan.host[:1024].view(np.int32)[164 + (M > 8)])
        assert (groups > 0) == (group is None)
        status = torch.full((B,), -1, dtype=torch.int32, device="cuda")
        doa.doa_solve_batch(plan, doa.workspace(plan), status)
        torch.cuda.synchronize()
        assert int(status.abs().max()) == 0
        assert bool((P[:, -1] == -1.0).all())       # nothing past a spectrum's end
        out.append((P, idx, val, cnt))
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("M", [5, 8, 13, 16])
def test_points_per_thread_give_the_same_spectrum(env, M):
    """A few scans take one point per thread (ULA and geometry, single calls and the batch): bit for bit
    the spectrum of four points per thread, at sizes on both sides of the rule."""
    torch, doa = env
    rng = np.random.default_rng(M)
    N = 128
    X = torch.view_as_complex(torch.randn(M, N, 2, generator=torch.Generator(device="cuda").manual_seed(M),
                                          device="cuda"))
    t = 2.0 * np.pi * np.arange(M) / M
    pos = torch.from_numpy(np.stack([0.5 * np.cos(t), 0.5 * np.sin(t), 0.1 * rng.standard_normal(M)], axis=1)).cuda()
    Q, _ = np.linalg.qr(rng.standard_normal((M, M)) + 1j * rng.standard_normal((M, M)))
    B = torch.from_numpy(np.ascontiguousarray(Q[:, :M - 2].T).reshape(-1)).cuda()
    for La, Le in ((1, 1), (97, 13), (360, 90), (361, 333)):
        out = []
        for pt in (None, (4, 4, 1, 1), (2, 2, 1, 1), (1, 1, 1, 1)):
            P = torch.zeros(4 * La * Le, device="cuda")
            idx = torch.full((8,), -1, dtype=torch.int32, device="cuda")
            val = torch.zeros(8, device="cuda")
            cnt = torch.zeros(4, dtype=torch.int32, device="cuda")
            prob = doa.make_problem(X, 2, 0xF, doa.grid(0.0, 360.0 / La, La), P, idx, val, cnt, None,
                                    geom=doa.geometry(pos, 2.0, 0.9, Le, True))
            plan = doa.BatchPlan([prob], scan_pt=pt)
            status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
            doa.doa_solve_batch(plan, doa.workspace(plan), status)
            torch.cuda.synchronize()
            assert int(status) == 0
            out.append((P, idx, val, cnt))
        for o in out[1:]:
            for a, b in zip(out[0], o):
                assert torch.equal(a, b)
    # single ULA scans: a long grid (four points per thread) against its pieces (one point per thread)
    L, piece = 100003, 7001
    P = torch.empty(L, device="cuda")
    doa.doa_scan(B, M, M - 2, doa.grid(-90.0, 180.0 / (L - 1), L), P)
    short = torch.empty(piece, device="cuda")
    doa.doa_scan(B, M, M - 2, doa.grid(-90.0, 180.0 / (L - 1), piece), short)
    torch.cuda.synchronize()
    assert torch.equal(P[:piece], short)
