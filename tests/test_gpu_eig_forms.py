"""The Jacobi's CTA form against its warp form and the oracle, at the sizes where the block folding and the
padding of odd M can go wrong."""
import numpy as np
import pytest

import oracle
from paper_2007_14135_gb300 import synth
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _solve(torch, doa, insts, prec, eig_mats):
    outs, probs = [], []
    for inst in insts:
        X = torch.from_numpy(inst.X).cuda()
        P = torch.empty(inst.L, dtype=torch.float32, device="cuda")
        idx = torch.full((max(inst.d, 1),), -1, dtype=torch.int32, device="cuda")
        val = torch.zeros(max(inst.d, 1), dtype=torch.float32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        ev = torch.zeros(inst.M, dtype=torch.float64, device="cuda")
        B = torch.zeros(inst.M * inst.M, dtype=torch.complex128, device="cuda")
        probs.append(doa.make_problem(X, inst.d, 1 << doa.MUSIC, doa.grid(inst.lo, inst.step, inst.L), P, idx, val, cnt,
                                      evals=ev, B_out=B, eig_prec=prec))
        outs.append((X, P, ev, B, idx, val, cnt))
    plan = doa.BatchPlan(probs, eig_mats=eig_mats)
    status = torch.full((len(insts),), -1, dtype=torch.int32, device="cuda")
    doa.doa_solve_batch(plan, doa.workspace(plan), status)
    torch.cuda.synchronize()
    assert status.cpu().numpy().tolist() == [0] * len(insts)
    return [(o[1].cpu().numpy(), o[2].cpu().numpy(), o[3].cpu().numpy()) for o in outs]


@pytest.mark.parametrize("prec", [0, 1])
def test_cta_and_warp_forms_agree_bit_for_bit(prec):
    """The same plan with a matrix per CTA (default for a small batch) and with packed warps."""
    torch, doa = require_gpu()
    insts = [synth.custom(M, max(1, M // 4), 200, None, 10.0, 1.0, seed=700 + M) for M in (2, 3, 5, 7, 8, 9, 11, 15, 16)]
    cta = _solve(torch, doa, insts, prec, [1, 1, 1, 1])
    warp = _solve(torch, doa, insts, prec, [2, 2, 1, 1])
    for a, b in zip(cta, warp):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("M", [2, 3, 5, 9, 13, 16, 17, 31, 32, 33, 63, 64])
@pytest.mark.parametrize("prec", [0, 1])
def test_single_calls_at_odd_sizes(M, prec):
    """Eigenvalues and C = B B^H of a single call against the oracle: 1e-12 of the largest in FP64; in
    double-float (2^-48 arithmetic, threshold 1e-12) 1e-10."""
    torch, doa = require_gpu()
    d = max(1, M // 4)
    R = oracle.covariance(synth.custom(M, d, 4 * M + 50, None, 10.0, 1.0, seed=800 + M).X)
    ev = torch.empty(M, dtype=torch.float64, device="cuda")
    B = torch.zeros(M * M, dtype=torch.complex128, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    doa.doa_noise_subspace_prec(torch.from_numpy(R).cuda(), d, doa.MUSIC, prec, B, info, evals=ev)
    torch.cuda.synchronize()
    assert info.item() > 0
    w, V = np.linalg.eigh(R)
    tol = 1e-12 if prec == doa.EIG_FP64 else 1e-10
    assert np.abs(ev.cpu().numpy() - w[::-1]).max() <= tol * w[-1]
    F = B.cpu().numpy()[:(M - d) * M].reshape(M - d, M).T
    E = V[:, :M - d]
    assert np.abs(F @ F.conj().T - E @ E.conj().T).max() <= 100 * tol


@pytest.mark.parametrize("M", [5, 9, 12, 16, 17, 31, 33])
@pytest.mark.parametrize("prec", [0, 1])
def test_digits_do_not_depend_on_the_outputs_asked_for(M, prec):
    """A geometry problem with and without peak_angle, in a CTA per matrix and packed: eigenvalues, factor and
    spectrum bit for bit (both halves of A are computed for either)."""
    torch, doa = require_gpu()
    rng = np.random.default_rng(900 + M)
    a = 2.0 * np.pi * np.arange(M) / M
    pos = np.stack([0.6 * np.cos(a), 0.6 * np.sin(a), np.zeros(M)], axis=1)
    X = torch.from_numpy((rng.standard_normal((M, 300)) + 1j * rng.standard_normal((M, 300))).astype(np.complex64)).cuda()
    posd, geom_grid = torch.from_numpy(pos).cuda(), doa.grid(0.0, 4.0, 90)
    geom = doa.geometry(posd, 2.0, 4.0, 20, True)
    results = []
    for refine, mats in ((False, None), (True, None), (True, [2, 2, 0, 0])):
        P = torch.zeros(90 * 20, dtype=torch.float32, device="cuda")
        idx = torch.full((2,), -1, dtype=torch.int32, device="cuda")
        val = torch.zeros(2, dtype=torch.float32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        ev = torch.zeros(M, dtype=torch.float64, device="cuda")
        B = torch.zeros(M * M, dtype=torch.complex128, device="cuda")
        ang = torch.zeros(4, dtype=torch.float64, device="cuda")
        plan = doa.BatchPlan([doa.make_problem(X, 2, 1 << doa.MUSIC, geom_grid, P, idx, val, cnt, evals=ev, B_out=B, geom=geom,
                                               eig_prec=prec, peak_angle=ang if refine else None)],
                             eig_mats=mats)
        status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        doa.doa_solve_batch(plan, doa.workspace(plan), status)
        torch.cuda.synchronize()
        assert status.item() == 0
        results.append((ev.cpu().numpy(), B.cpu().numpy(), P.cpu().numpy()))
    for r in results[1:]:
        for x, y in zip(results[0], r):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("M", [7, 13, 16, 24, 32])
def test_digits_do_not_depend_on_the_neighbours_arithmetic(M):
    """A bucket with an FP64 problem takes FP64's CTA size: the double-float problems' outputs, and the FP64 one's,
    are those of buckets of one arithmetic."""
    torch, doa = require_gpu()
    insts = [synth.custom(M, max(1, M // 4), 200, None, 10.0, 1.0, seed=960 + M + i) for i in range(3)]

    def solve(precs):
        outs, probs = [], []
        for inst, prec in zip(insts, precs):
            X = torch.from_numpy(inst.X).cuda()
            P = torch.empty(inst.L, dtype=torch.float32, device="cuda")
            pk = [torch.zeros(inst.d, dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
            cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
            ev = torch.zeros(M, dtype=torch.float64, device="cuda")
            B = torch.zeros(M * M, dtype=torch.complex128, device="cuda")
            probs.append(doa.make_problem(X, inst.d, 1 << doa.MUSIC, doa.grid(inst.lo, inst.step, inst.L), P, *pk, cnt,
                                          evals=ev, B_out=B, eig_prec=prec))
            outs.append((X, P, ev, B, pk, cnt))
        status = torch.full((len(insts),), -1, dtype=torch.int32, device="cuda")
        plan = doa.BatchPlan(probs)
        doa.doa_solve_batch(plan, doa.workspace(plan), status)
        torch.cuda.synchronize()
        assert status.cpu().tolist() == [0] * len(insts)
        return [[t.cpu().numpy() for t in o[1:4]] for o in outs]

    df, f64 = doa.EIG_DOUBLE_FLOAT, doa.EIG_FP64
    mixed, alone, wide = solve([df, f64, df]), solve([df, df, df]), solve([f64, f64, f64])
    for got, want in zip(mixed, (alone[0], wide[1], alone[2])):
        for x, y in zip(got, want):
            np.testing.assert_array_equal(x, y)
