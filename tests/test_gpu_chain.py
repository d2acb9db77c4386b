"""Calls that follow one another in a stream without a synchronisation: the kernels of a chain are queued
behind each other (some start beside the one before), and new inputs go into the same buffers while the
last results are still being computed. Results are those of the same calls one at a time, bit for bit,
directly and from a captured graph."""
import numpy as np
import pytest

from tests.gpu_common import MUSIC, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return require_gpu()


def _inputs(torch, n, shape, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda")) for _ in range(n)]


@pytest.mark.parametrize("M,N,L,fp64", [(5, 100, 181, True), (8, 1024, 1801, True), (16, 2048, 18001, False),
                                        (33, 600, 1801, False), (64, 4096, 100001, False)])
def test_single_calls(env, M, N, L, fp64):
    torch, doa = env
    d, n = 2, 6
    Xs = _inputs(torch, n, (M, N), M)
    X, g = torch.empty_like(Xs[0]), doa.grid(-90.0, 180.0 / (L - 1), L)
    R = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
    B = torch.zeros(M * M, dtype=torch.complex128, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    P = torch.zeros(L, device="cuda")
    idx = torch.full((d,), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(d, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    outs = (R, B, P, idx, val, cnt)

    def chain(sync):
        pause = torch.cuda.synchronize if sync else (lambda: None)
        doa.doa_covariance(X, R64=R)
        pause()
        doa.doa_noise_subspace_prec(R, d, MUSIC, doa.EIG_FP64 if fp64 else doa.EIG_DOUBLE_FLOAT, B, info)
        pause()
        doa.doa_scan(B, M, M - d, g, P)
        pause()
        doa.doa_peaks(P, d, idx, val, cnt)
        pause()

    want = []
    for x in Xs:
        X.copy_(x)
        chain(True)
        want.append([o.clone() for o in outs])
    got = []
    for x in Xs:
        X.copy_(x)
        chain(False)
        got.append([o.clone() for o in outs])
    torch.cuda.synchronize()
    for w, o in zip(want, got):
        for a, b in zip(w, o):
            assert torch.equal(a, b)


@pytest.mark.parametrize("Ms,geo", [((8,), False), ((8, 16), True), ((3, 12, 31, 50), True), ((16, 24, 64), False)])
@pytest.mark.parametrize("B", [1, 40])
def test_batch_solves(env, Ms, geo, B):
    torch, doa = env
    d, N, n, L = 1, 301, 5, 1801
    t = 2.0 * np.pi * np.arange(8) / 8
    pos = torch.from_numpy(np.stack([0.5 * np.sin(t), 0.5 * np.cos(t), 0 * t], axis=1)).cuda()
    shapes = [(M, False) for M in Ms for _ in range(B)] + ([(8, True)] * B if geo else [])
    Xs = [_inputs(torch, n, (M, N + (i % 2)), 10 * i + M) for i, (M, _) in enumerate(shapes)]
    X, outs, probs = [x[0].clone() for x in Xs], [], []
    for x, (M, is_geo) in zip(X, shapes):
        npts = 360 * 10 if is_geo else L
        o = (torch.zeros(4 * npts, device="cuda"), torch.full((4 * d,), -1, dtype=torch.int32, device="cuda"),
             torch.zeros(4 * d, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda"),
             torch.zeros(M, dtype=torch.float64, device="cuda"))
        outs.append(o)
        if is_geo:
            probs.append(doa.make_problem(x, d, 0xF, doa.grid(0.0, 1.0, 360), *o,
                                          geom=doa.geometry(pos, 1.0, 9.0, 10, True)))
        else:
            probs.append(doa.make_problem(x, d, 0xF, doa.grid(-90.0, 0.1, L), *o, polish=True))
    plan = doa.BatchPlan(probs)
    ws = doa.workspace(plan)
    status = torch.full((len(probs),), -1, dtype=torch.int32, device="cuda")

    def fill(k):
        for x, xs in zip(X, Xs):
            x.copy_(xs[k])

    want = []
    for k in range(n):
        fill(k)
        torch.cuda.synchronize()
        doa.doa_solve_batch(plan, ws, status)
        torch.cuda.synchronize()
        assert int(status.abs().max()) == 0
        want.append([[a.clone() for a in o] for o in outs])
    got = []
    for k in range(n):
        fill(k)
        doa.doa_solve_batch(plan, ws, status)
        got.append([[a.clone() for a in o] for o in outs])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        doa.doa_solve_batch(plan, ws, status, stream=s)
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        doa.doa_solve_batch(plan, ws, status)
    for k in range(n):
        fill(k)
        g.replay()
        got.append([[a.clone() for a in o] for o in outs])
    torch.cuda.synchronize()
    for w, res in zip(want + want, got):
        for a, b in zip(w, res):
            for p, q in zip(a, b):
                assert torch.equal(p, q)
