"""What is measured when this library is timed: calls of its public entry points as users make them.

listed() gives the cases, draw(rng) more of the same ranges. prepare(case, seed) makes on the GPU what a
program has in hand before the call (snapshots, output buffers, the plan and workspace it keeps, the
network), run(state) makes the call and returns everything it computes, exact(case, seed) computes the same
in 64 bits with plain torch / numpy, and work(case) is what the method itself has to read, write and compute.

Kinds of case:
  chain      one estimate by single calls: covariance, eigendecomposition, scan, peaks
  batch      many ULA problems in one plan, all of one shape
  uneven     many ULA problems of mixed M, d, N, grid and algorithm in one plan
  circle     azimuth x elevation scans of a circular array in one plan
  estimates  a plan that asks for every estimate: refined angles, polynomial roots, model order; ULA and circle
  svd        Step-2 as a one-sided Jacobi SVD of the snapshots
  forward    the proposal network's forward pass
  train      one training step of the proposal network (gradients, then Adam)
  windows    the learned proposal's decode, windowed fine scan and judge
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2007_14135_gb300 import doa

DEV = "cuda"
PHD, MUSIC, EV, MN = 0, 1, 2, 3
FP32, BF16X3, FP16X3 = doa.FP32, doa.BF16X3, doa.FP16X3
C64, C128, F32, F64, I32 = torch.complex64, torch.complex128, torch.float32, torch.float64, torch.int32
UCA_RADIUS = 10.0 * 15e6 / 299792458.0      # 10 m at 15 MHz, in wavelengths
NET = (272, 256, 256, 256, 181)


def grid_size(step):
    return int(round(180.0 / step)) + 1


def listed():
    return [
        # one small estimate, as a receiver makes it again and again: latency and launches
        {"name": "one_m8", "kind": "chain", "M": 8, "N": 1024, "d": 2, "step": 0.1, "alg": MUSIC, "prec": FP32, "fp64": True},
        # one estimate of a large array on a very fine grid, the split-precision scan
        {"name": "one_m64", "kind": "chain", "M": 64, "N": 16384, "d": 8, "step": 0.0005, "alg": MUSIC, "prec": FP16X3,
         "fp64": False},
        # the paper's own scenario: one circular-array estimate on the 360 x 90 scan
        {"name": "one_circle", "kind": "circle", "B": 1, "M": 8, "N": 1024, "d": 2, "La": 360, "Le": 90, "refine": False},
        # the paper-density batch, all four algorithms, as a server solves it
        {"name": "batch_m16", "kind": "batch", "B": 4096, "M": 16, "N": 4096, "d": 4, "step": 0.01, "mask": 15, "prec": FP32,
         "fp64": False, "polish": True},
        # mixed requests in one plan
        {"name": "batch_uneven", "kind": "uneven", "B": 1024, "odd": False, "nmax": 8192, "mix": 1},
        # many circular-array estimates
        {"name": "batch_circle", "kind": "circle", "B": 4096, "M": 8, "N": 1024, "d": 2, "La": 360, "Le": 90, "refine": False},
        # off-grid estimates: refinement, root form and model order beside the peaks
        {"name": "estimates", "kind": "estimates", "B": 512, "M": 16, "N": 2048, "d": 4, "step": 0.1, "circles": 512},
        # Step-2 as an SVD, at the paper-density size and at the largest array
        {"name": "svd_m16", "kind": "svd", "M": 16, "N": 4096, "d": 4, "c128": False},
        {"name": "svd_m64", "kind": "svd", "M": 64, "N": 16384, "d": 8, "c128": False},
        # the proposal network on a test set, and one step of its training
        {"name": "net_forward", "kind": "forward", "B": 65536},
        {"name": "net_train", "kind": "train", "B": 4096},
        # the learned proposal's fine scan: windows of +-2 degrees at 0.001 degree, and the judge
        {"name": "windows", "kind": "windows", "B": 2048, "d": 4, "width": 4001},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "batch", "batch", "uneven", "uneven", "circle", "circle", "estimates", "svd", "svd",
                       "forward", "train", "windows"])
    if kind == "chain":
        M = _log(rng, 4, 64)
        prec = rng.choice([FP32, FP32, BF16X3, FP16X3])
        N = _log(rng, 64, 16384)
        if prec != FP32:
            N += N % 2          # the tensor-core covariance reads rows of an even stride
        return {"kind": kind, "M": M, "N": N, "d": rng.randint(1, max(1, M // 4)),
                "step": rng.choice([1.0, 0.1, 0.01, 0.001]), "alg": rng.choice([MUSIC, EV]), "prec": prec,
                "fp64": M <= 16 or rng.random() < 0.3}
    if kind == "batch":
        M = rng.choice([4, 7, 8, 12, 13, 16, 16, 24, 32])
        return {"kind": kind, "B": _log(rng, 1, 4096 if M <= 16 else 512), "M": M, "N": _log(rng, 128, 4096),
                "d": rng.randint(1, max(1, M // 4)), "step": rng.choice([1.0, 0.1, 0.01]),
                "mask": rng.choice([1 << MUSIC, 1 << EV, 1 << PHD, 1 << MUSIC | 1 << MN, 15]),
                "prec": rng.choice([FP32, FP32, FP16X3, BF16X3]), "fp64": rng.random() < 0.2, "polish": True}
    if kind == "uneven":
        return {"kind": kind, "B": _log(rng, 64, 1024), "odd": rng.random() < 0.5, "nmax": _log(rng, 512, 8192), "mix": rng.randint(2, 1 << 30)}
    if kind == "circle":
        return {"kind": kind, "B": _log(rng, 1, 4096), "M": rng.choice([5, 8, 8, 12, 16]), "N": _log(rng, 128, 1024), "d": 2,
                "La": rng.choice([180, 360, 360, 361]), "Le": rng.randint(1, 90), "refine": rng.random() < 0.3}
    if kind == "estimates":
        M = rng.choice([6, 8, 11, 16, 20])
        return {"kind": kind, "B": _log(rng, 16, 512), "M": M, "N": _log(rng, 256, 2048), "d": rng.randint(1, M // 4),
                "step": rng.choice([0.5, 0.1]), "circles": _log(rng, 1, 512)}
    if kind == "svd":
        M = _log(rng, 4, 48)
        return {"kind": kind, "M": M, "N": _log(rng, 128, 8192), "d": max(1, M // 8), "c128": rng.random() < 0.3}
    if kind == "forward":
        return {"kind": kind, "B": 8 * _log(rng, 1, 8192)}
    if kind == "train":
        return {"kind": kind, "B": 8 * _log(rng, 16, 1024)}
    return {"kind": "windows", "B": _log(rng, 64, 2048), "d": rng.randint(1, 6), "width": rng.choice([2001, 4001])}


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    """CN(0, 1) samples, complex64."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV) * math.sqrt(0.5))


def _angles(rng, B, d, lo, hi, sep):
    """(B, d) ascending angles in [lo, hi], at least sep apart."""
    sep = min(sep, 0.5 * (hi - lo) / d)
    u = np.sort(rng.uniform(0.0, (hi - lo) - (d - 1) * sep, size=(B, d)), axis=1)
    return lo + u + sep * np.arange(d)[None, :]


def _mix(g, A, N, snr_db):
    """X = A S + W for responses A (B, M, d) and one SNR per row, complex64 (B, M, N)."""
    B, M, d = A.shape
    A = torch.from_numpy(A.astype(np.complex64)).to(DEV)
    sigma = torch.from_numpy((10.0 ** (-snr_db / 20.0)).astype(np.float32)).to(DEV)
    X = torch.empty((B, M, N), dtype=C64, device=DEV)
    for s in range(0, B, 512):
        e = min(B, s + 512)
        X[s:e] = torch.bmm(A[s:e], _randn(g, e - s, d, N)) + sigma[s:e, None, None] * _randn(g, e - s, M, N)
    return X


def _ula_snapshots(seed, B, M, N, d, sep, snr):
    """Snapshots of B uniform linear arrays: d unit-power sources in +-60 degrees, white noise."""
    rng = np.random.default_rng([seed, M, N, d])
    ang = _angles(rng, B, d, -60.0, 60.0, sep)
    A = np.exp(1j * np.pi * np.arange(M)[None, :, None] * np.sin(np.deg2rad(ang))[:, None, :])
    return _mix(_gen(seed), A, N, rng.uniform(*snr, size=B))


def _circle_positions(M):
    a = 2.0 * np.pi * np.arange(M) / M
    return np.stack([UCA_RADIUS * np.sin(a), UCA_RADIUS * np.cos(a), np.zeros(M)], axis=1)


def _circle_snapshots(seed, B, M, N, d):
    rng = np.random.default_rng([seed, M, N, d, 1])
    az = rng.uniform(0.0, 360.0, size=(B, 1)) + np.concatenate([np.zeros((B, 1)), rng.uniform(30.0, 330.0, size=(B, d - 1))], axis=1)
    el = np.deg2rad(rng.uniform(10.0, 90.0, size=(B, d)))
    az = np.deg2rad(az)
    u = np.stack([np.sin(az) * np.sin(el), np.cos(az) * np.sin(el), np.cos(el)], axis=1)     # (B, 3, d)
    A = np.exp(2j * np.pi * np.einsum("mx,bxd->bmd", _circle_positions(M), u))
    return _mix(_gen(seed), A, N, np.full(B, 15.0))


def _uneven_specs(case):
    """M, d, N, grid step and algorithm of each problem, as requests of many users mix them."""
    rng = np.random.default_rng([case["mix"], case["B"]])
    sizes = [3, 5, 7, 8, 11, 12, 16, 23, 32, 48, 64] if case["odd"] else [8, 12, 16, 32]
    out = []
    for _ in range(case["B"]):
        M = int(rng.choice(sizes))
        out.append((M, int(rng.integers(1, M // 2 + 1)), int(rng.integers(min(256, case["nmax"] // 2), case["nmax"] + 1)),
                    float(rng.choice([0.1, 0.01, 0.001])), int(rng.integers(0, 4))))
    return out


def _uneven_snapshots(case, seed, specs):
    """One flat buffer of all the problems' snapshots and each one's offset; rows are packed."""
    rng = np.random.default_rng([seed, case["B"], 1])
    g = _gen(seed)
    size = [M * N for M, d, N, step, alg in specs]
    offs = np.concatenate([[0], np.cumsum([(s + 31) // 32 * 32 for s in size])])
    buf = torch.zeros(int(offs[-1]), dtype=C64, device=DEV)
    for o, (M, d, N, step, alg) in zip(offs, specs):
        s = np.sin(np.deg2rad(_angles(rng, 1, d, -60.0, 60.0, 5.0)[0]))
        A = torch.from_numpy(np.exp(1j * np.pi * np.arange(M)[:, None] * s[None, :]).astype(np.complex64)).to(DEV)
        sigma = 10.0 ** (-rng.uniform(0.0, 20.0) / 20.0)
        buf[int(o):int(o) + M * N] = (A @ _randn(g, d, N) + sigma * _randn(g, M, N)).reshape(-1)
    return buf, offs


# ------------------------------------------------------------------------------------------------ prepare
def _solver(problems, nprob):
    plan = doa.BatchPlan(problems, device=DEV)
    return {"plan": plan, "ws": doa.workspace(plan, device=DEV), "status": torch.zeros(nprob, dtype=I32, device=DEV)}


def _peak_buffers(B, nalg, d):
    return {"idx": torch.full((B, nalg, d), -1, dtype=I32, device=DEV), "val": torch.zeros((B, nalg, d), dtype=F32, device=DEV),
            "cnt": torch.zeros((B, nalg), dtype=I32, device=DEV)}


def _prepare_chain(case, seed):
    M, d, L = case["M"], case["d"], grid_size(case["step"])
    fac = torch.zeros(M * M, dtype=C128, device=DEV)          # the entry point asks for room for M x M
    o = {"R": torch.zeros((M, M), dtype=C128, device=DEV), "evals": torch.zeros(M, dtype=F64, device=DEV),
         "B": fac[:(M - d) * M], "P": torch.zeros(L, dtype=F32, device=DEV),
         "idx": torch.full((d,), -1, dtype=I32, device=DEV), "val": torch.zeros(d, dtype=F32, device=DEV),
         "cnt": torch.zeros(1, dtype=I32, device=DEV), "info": torch.zeros(1, dtype=I32, device=DEV)}
    return {"case": case, "X": _ula_snapshots(seed, 1, M, case["N"], d, 1.0 if M > 32 else 5.0, (0.0, 15.0))[0], "fac": fac,
            "out": o, "grid": doa.grid(-90.0, case["step"], L)}


def _prepare_batch(case, seed):
    B, M, d, mask = case["B"], case["M"], case["d"], case["mask"]
    nalg, L = bin(mask).count("1"), grid_size(case["step"])
    X = _ula_snapshots(seed, B, M, case["N"], d, 5.0, (0.0, 20.0))
    o = {"P": torch.zeros((B, nalg, L), dtype=F32, device=DEV), "evals": torch.zeros((B, M), dtype=F64, device=DEV),
         **_peak_buffers(B, nalg, d)}
    g = doa.grid(-90.0, case["step"], L)
    probs = [doa.make_problem(X[i], d, mask, g, o["P"][i], o["idx"][i], o["val"][i], o["cnt"][i], evals=o["evals"][i],
                              prec=case["prec"], eig_prec=doa.EIG_FP64 if case["fp64"] else doa.EIG_DOUBLE_FLOAT,
                              polish=case["polish"]) for i in range(B)]
    return {"case": case, "X": X, "out": o, **_solver(probs, B)}


def _prepare_uneven(case, seed):
    specs = _uneven_specs(case)
    buf, offs = _uneven_snapshots(case, seed, specs)
    Ls = [grid_size(s[3]) for s in specs]
    po = np.concatenate([[0], np.cumsum(Ls)])
    dmax = max(s[1] for s in specs)
    o = {"P": torch.zeros(int(po[-1]), dtype=F32, device=DEV), **_peak_buffers(len(specs), 1, dmax),
         "evals": torch.zeros((len(specs), 64), dtype=F64, device=DEV)}
    probs = []
    for i, (M, d, N, step, alg) in enumerate(specs):
        X = buf[int(offs[i]):int(offs[i]) + M * N].view(M, N)
        probs.append(doa.make_problem(X, d, 1 << alg, doa.grid(-90.0, step, Ls[i]), o["P"][int(po[i]):int(po[i + 1])],
                                      o["idx"][i, 0], o["val"][i, 0], o["cnt"][i], evals=o["evals"][i], polish=True))
    return {"case": case, "X": buf, "out": o, **_solver(probs, len(specs))}


def _circle_problems(case, X, pos, o):
    B = X.shape[0]
    geom = doa.geometry(pos, float(91 - case["Le"]), 1.0, case["Le"], case["La"] == 360)
    g = doa.grid(0.0, 2.0 if case["La"] == 180 else 1.0, case["La"])
    return [doa.make_problem(X[i], case["d"], 1 << MUSIC, g, o["P"][i], o["idx"][i], o["val"][i], o["cnt"][i],
                             evals=o["evals"][i], geom=geom, peak_angle=o["angle"][i] if "angle" in o else None) for i in range(B)]


def _circle_buffers(B, case, refine):
    o = {"P": torch.zeros((B, case["Le"], case["La"]), dtype=F32, device=DEV), **_peak_buffers(B, 1, case["d"]),
         "evals": torch.zeros((B, case["M"]), dtype=F64, device=DEV)}
    if refine:
        o["angle"] = torch.zeros((B, 1, case["d"], 2), dtype=F64, device=DEV)
    return o


def _prepare_circle(case, seed):
    B = case["B"]
    X = _circle_snapshots(seed, B, case["M"], case["N"], case["d"])
    pos = torch.from_numpy(_circle_positions(case["M"])).to(DEV)
    o = _circle_buffers(B, case, case["refine"])
    return {"case": case, "X": X, "pos": pos, "out": o, **_solver(_circle_problems(case, X, pos, o), B)}


def _estimate_circle(case):
    return {"M": 8, "N": 1024, "d": 2, "La": 360, "Le": 45}


def _prepare_estimates(case, seed):
    B, M, d, nc = case["B"], case["M"], case["d"], case["circles"]
    L = grid_size(case["step"])
    X = _ula_snapshots(seed, B, M, case["N"], d, 8.0, (5.0, 20.0))
    o = {"P": torch.zeros((B, 4, L), dtype=F32, device=DEV), "evals": torch.zeros((B, M), dtype=F64, device=DEV),
         **_peak_buffers(B, 4, d), "angle": torch.zeros((B, 4, d), dtype=F64, device=DEV),
         "order": torch.zeros((B, 2), dtype=I32, device=DEV), "root": torch.zeros((B, 4, d), dtype=F64, device=DEV)}
    g = doa.grid(-90.0, case["step"], L)
    probs = [doa.make_problem(X[i], d, 15, g, o["P"][i], o["idx"][i], o["val"][i], o["cnt"][i], evals=o["evals"][i], polish=True,
                              peak_angle=o["angle"][i], order_est=o["order"][i], root_angle=o["root"][i]) for i in range(B)]
    cc = _estimate_circle(case)
    Xc = _circle_snapshots(seed, nc, cc["M"], cc["N"], cc["d"])
    pos = torch.from_numpy(_circle_positions(cc["M"])).to(DEV)
    oc = _circle_buffers(nc, cc, True)
    probs += _circle_problems(cc, Xc, pos, oc)
    return {"case": case, "X": (X, Xc), "pos": pos, "out": {"ula": o, "circle": oc}, **_solver(probs, B + nc)}


def _svd_snapshots(case, seed):
    X = _ula_snapshots(seed, 1, case["M"], case["N"], case["d"], 5.0, (0.0, 20.0))[0]
    return X.to(C128) if case["c128"] else X


def _prepare_svd(case, seed):
    M, N = case["M"], case["N"]
    return {"case": case, "X": _svd_snapshots(case, seed), "ws": torch.zeros(max(doa.svd_data_ws_bytes(M, N), 256), dtype=torch.uint8, device=DEV),
            "out": {"evals": torch.zeros(M, dtype=F64, device=DEV), "U": torch.zeros((M, M), dtype=C128, device=DEV),
                    "info": torch.zeros(1, dtype=I32, device=DEV)}}


def _features(seed, B):
    """The network's input: the upper triangle of trace-normalised covariances (M = 16, up to six sources)."""
    g = _gen(seed)
    M = 16
    iu = torch.triu_indices(M, M, device=DEV)
    out = torch.empty((B, M * (M + 1)), dtype=F32, device=DEV)
    m = torch.arange(M, device=DEV, dtype=F32)
    for s in range(0, B, 8192):
        n = min(B, s + 8192) - s
        ang = torch.deg2rad(torch.rand(n, 6, generator=g, device=DEV) * 160.0 - 80.0)
        p = (torch.rand(n, 6, generator=g, device=DEV) < 0.6).float()
        ph = math.pi * m[None, :, None] * torch.sin(ang)[:, None, :]
        A = torch.polar(torch.ones_like(ph), ph)
        noise = 10.0 ** (-(torch.rand(n, 1, 1, generator=g, device=DEV) * 25.0 - 5.0) / 10.0)
        W = _randn(g, n, M, 256)
        R = torch.bmm(A * p[:, None, :], A.mH) + noise * torch.bmm(W, W.mH) / 256.0
        R = R / torch.diagonal(R, dim1=1, dim2=2).real.sum(1)[:, None, None]
        out[s:s + n] = torch.view_as_real(R[:, iu[0], iu[1]]).reshape(n, -1)
    return out


def _net(seed):
    """A network some way into its training: weights of its initial scale, biases and Adam moments not zero."""
    net = doa.Mlp(seed=seed % 1000003, device=DEV)
    g = _gen(seed + 1)
    for l in range(4):
        net.buf["b"][l].copy_(0.05 * torch.randn(NET[l + 1], generator=g, device=DEV))
        for m, v in (("mW", "vW"), ("mb", "vb")):
            net.buf[m][l].copy_(1e-3 * torch.randn(net.buf[m][l].shape, generator=g, device=DEV))
            net.buf[v][l].copy_(1e-5 * (0.5 + torch.rand(net.buf[v][l].shape, generator=g, device=DEV)))
    net.t = 1000
    return net


def _labels(seed, B):
    return (torch.rand(B, NET[-1], generator=_gen(seed + 2), device=DEV) < 0.02).to(F32)


def _prepare_forward(case, seed):
    net, B = _net(seed), case["B"]
    return {"case": case, "net": net, "x": _features(seed, B), "ws": net.workspace(B),
            "out": {"probs": torch.zeros((B, NET[-1]), dtype=F32, device=DEV), "logits": torch.zeros((B, NET[-1]), dtype=F32, device=DEV)}}


def _prepare_train(case, seed):
    net, B = _net(seed), case["B"]
    return {"case": case, "net": net, "x": _features(seed, B), "y": _labels(seed, B), "ws": net.workspace(B),
            "loss": torch.zeros(1, dtype=F32, device=DEV)}


def _window_inputs(case, seed):
    """MUSIC factors, coarse spectra and occupancy probabilities (high near the sources) of B instances."""
    B, d, M = case["B"], case["d"], 16
    rng = np.random.default_rng([seed, B, d, 7])
    ang = _angles(rng, B, d, -75.0, 75.0, 6.0)
    A = np.exp(1j * np.pi * np.arange(M)[None, :, None] * np.sin(np.deg2rad(ang))[:, None, :])
    X = _mix(_gen(seed), A, 512, rng.uniform(0.0, 20.0, size=B)).to(C128)
    _, V = torch.linalg.eigh(torch.bmm(X, X.mH) / 512)         # ascending: the noise subspace comes first
    F = torch.zeros((B, M, M), dtype=C128, device=DEV)         # row k: column k of the factor
    F[:, :M - d] = V[:, :, :M - d].transpose(1, 2)
    th = torch.deg2rad(-90.0 + 0.1 * torch.arange(1801, device=DEV, dtype=F64))
    a = torch.polar(torch.ones(M, 1801, dtype=F64, device=DEV), math.pi * torch.arange(M, device=DEV, dtype=F64)[:, None] * torch.sin(th)[None, :])
    Pc = torch.cat([1.0 / (torch.matmul(F[s:s + 256, :M - d].conj(), a).abs() ** 2).sum(1) for s in range(0, B, 256)]).to(F32)
    probs = 0.05 * torch.rand(B, 181, generator=_gen(seed + 3), device=DEV)
    bins = torch.from_numpy(np.rint(ang).astype(np.int64) + 90).to(DEV)
    probs.scatter_(1, bins, 0.5 + 0.45 * torch.rand(B, d, generator=_gen(seed + 4), device=DEV))
    return F, Pc, probs


def _prepare_windows(case, seed):
    B, w = case["B"], case["width"]
    F, Pc, probs = _window_inputs(case, seed)
    fine = doa.grid(-90.0, 0.001, 180001)
    o = {"win": torch.full((B, 8), -1, dtype=I32, device=DEV), "idx": torch.full((B, 8), -1, dtype=I32, device=DEV),
         "val": torch.zeros((B, 8), dtype=F32, device=DEV), "cnt": torch.zeros(B, dtype=I32, device=DEV),
         "fallback": torch.zeros(B, dtype=I32, device=DEV), "judge": torch.full((B, doa.JUDGE_MAX), -1, dtype=I32, device=DEV),
         "spectra": torch.zeros((B, 8, w), dtype=F32, device=DEV)}
    return {"case": case, "B": F.reshape(B, -1), "Pc": Pc, "probs": probs, "fine": fine, "coarse": doa.grid(-90.0, 0.1, 1801), "out": o,
            "d": torch.full((B,), case["d"], dtype=I32, device=DEV), "K": torch.full((B,), 16 - case["d"], dtype=I32, device=DEV),
            "S": torch.zeros(fine.L, dtype=I32, device=DEV), "Pj": torch.zeros((B, doa.JUDGE_MAX, 401), dtype=F32, device=DEV)}


def prepare(case, seed):
    return {"chain": _prepare_chain, "batch": _prepare_batch, "uneven": _prepare_uneven, "circle": _prepare_circle,
            "estimates": _prepare_estimates, "svd": _prepare_svd, "forward": _prepare_forward, "train": _prepare_train,
            "windows": _prepare_windows}[case["kind"]](case, seed)


# ------------------------------------------------------------------------------------------------ run
def _run_chain(s):
    c, o, X = s["case"], s["out"], s["X"]
    M, d = c["M"], c["d"]
    doa.doa_covariance(X, R64=o["R"], prec=c["prec"])
    doa.doa_noise_subspace_prec(o["R"], d, c["alg"], doa.EIG_FP64 if c["fp64"] else doa.EIG_DOUBLE_FLOAT, s["fac"], o["info"],
                                evals=o["evals"])
    doa.doa_scan(s["fac"], M, M - d, s["grid"], o["P"], prec=c["prec"])
    doa.doa_peaks(o["P"], d, o["idx"], o["val"], o["cnt"])
    return {k: v for k, v in o.items() if k != "info"}


def _run_plan(s):
    doa.doa_solve_batch(s["plan"], s["ws"], s["status"])
    return {"status": s["status"], **s["out"]}


def _run_svd(s):
    o = s["out"]
    doa.doa_svd_data(s["X"], o["evals"], o["U"], o["info"], ws=s["ws"])
    return {"evals": o["evals"], "U": o["U"]}


def _run_forward(s):
    s["net"].forward(s["x"], s["ws"], probs=s["out"]["probs"], logits=s["out"]["logits"])
    return s["out"]


def _run_train(s):
    net = s["net"]
    net.backward(s["x"], s["y"], s["ws"], loss=s["loss"])
    net.adam(1e-4)
    return {"loss": s["loss"], **{k: list(net.buf[k]) for k in ("gW", "gb", "W", "b", "mW", "mb", "vW", "vb")}}


def _run_windows(s):
    c, o = s["case"], s["out"]
    doa.doa_proposal_windows(s["probs"], s["d"], s["fine"], c["width"], o["win"], extra=2)
    doa.doa_scan_windows(s["B"], 16, s["K"], s["d"], s["fine"], s["S"], o["spectra"], o["idx"], o["val"], o["cnt"],
                         win_first=o["win"], width=c["width"], fallback=o["fallback"])
    doa.doa_proposal_judge(s["B"], 16, s["K"], s["d"], s["Pc"], s["coarse"], s["fine"], o["win"], c["width"], o["val"], o["cnt"],
                           401, o["judge"], s["S"], s["Pj"], o["fallback"])
    return o


def run(state):
    kind = state["case"]["kind"]
    if kind in ("batch", "uneven", "circle", "estimates"):
        return _run_plan(state)
    return {"chain": _run_chain, "svd": _run_svd, "forward": _run_forward, "train": _run_train, "windows": _run_windows}[kind](state)


# ------------------------------------------------------------------------------------------------ work
def _cov_flops(M, N):
    return 4.0 * M * M * N               # one triangle of complex multiply-adds


def _eig_flops(M):
    return 40.0 * M ** 3                 # tridiagonalisation, QR and eigenvectors of a Hermitian matrix


def _scan_flops(M, d, mask):
    """Per point: y = F^H a for the columns the algorithms need, and their weighted norms."""
    cols = (M - d if mask & 6 else 1 if mask & 1 else 0) + (1 if mask & 8 else 0)
    return cols * 8.0 * M + 4.0 * cols * bin(mask).count("1")


def _problem_work(M, N, d, points, mask, prec=FP32):
    nalg = bin(mask).count("1")
    return {"bytes": 8.0 * M * N + 4.0 * nalg * points + 8.0 * M + 8.0 * nalg * d,
            "flops": _cov_flops(M, N) + _eig_flops(M) + points * _scan_flops(M, d, mask)}


def _sum(works):
    works = list(works)
    return {k: float(sum(w[k] for w in works)) for k in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "chain":
        w = _problem_work(case["M"], case["N"], case["d"], grid_size(case["step"]), 1 << case["alg"])
        return {"bytes": w["bytes"] + 16.0 * case["M"] ** 2, "flops": w["flops"]}
    if kind == "batch":
        w = _problem_work(case["M"], case["N"], case["d"], grid_size(case["step"]), case["mask"])
        return {k: v * case["B"] for k, v in w.items()}
    if kind == "uneven":
        return _sum(_problem_work(M, N, d, grid_size(step), 1 << alg) for M, d, N, step, alg in _uneven_specs(case))
    if kind == "circle":
        w = _problem_work(case["M"], case["N"], case["d"], case["La"] * case["Le"], 1 << MUSIC)
        return {k: v * case["B"] for k, v in w.items()}
    if kind == "estimates":
        cc = _estimate_circle(case)
        u = _problem_work(case["M"], case["N"], case["d"], grid_size(case["step"]), 15)
        # refinement: a few evaluations of den and its derivatives; roots: a few sweeps over the 2M - 2 roots
        u["flops"] += 4 * case["d"] * 5 * 16.0 * case["M"] ** 2 + 4 * 10 * 24.0 * (2 * case["M"] - 2) ** 2
        v = _problem_work(cc["M"], cc["N"], cc["d"], cc["La"] * cc["Le"], 1 << MUSIC)
        v["flops"] += cc["d"] * 5 * 40.0 * cc["M"] ** 2
        return {k: u[k] * case["B"] + v[k] * case["circles"] for k in u}
    if kind == "svd":
        M, N = case["M"], case["N"]
        return {"bytes": (16.0 if case["c128"] else 8.0) * M * N + 16.0 * M * M, "flops": _cov_flops(M, N) + _eig_flops(M)}
    params = float(sum(NET[l] * NET[l + 1] for l in range(4)))
    if kind == "forward":
        return {"bytes": case["B"] * (NET[0] + 2 * NET[-1]) * 4.0 + params * 2, "flops": 2.0 * params * case["B"]}
    if kind == "train":
        return {"bytes": case["B"] * (NET[0] + NET[-1]) * 4.0 + params * 28, "flops": 6.0 * params * case["B"]}
    points = float(case["B"]) * (case["d"] + 2) * case["width"]
    return {"bytes": 4.0 * points + case["B"] * (16.0 * 16 * (16 - case["d"]) + 4.0 * (1801 + 181)),
            "flops": points * _scan_flops(16, case["d"], 1 << MUSIC)}


# ------------------------------------------------------------------------------------------------ exact
def _covariance(X):
    X = X.to(C128)
    return X @ X.mH / X.shape[-1]


def _subspace(R):
    """Eigenvalues and eigenvectors (columns), descending."""
    w, V = torch.linalg.eigh(R)
    return w.flip(-1), V.flip(-1)


def _factor(w, V, d, alg):
    """B with C = B B^H (Table 3), columns last; w (..., M), V (..., M, M)."""
    if alg == PHD:
        return V[..., -1:]
    E = V[..., d:]
    if alg == MUSIC:
        return E
    if alg == EV:
        return E * (1.0 / torch.sqrt(w[..., None, d:]))
    p = E @ E[..., :1, :].mH                                  # P_n e1
    return p / p[..., :1, :].real


def _ula_steering(M, th):
    ph = math.pi * torch.arange(M, device=DEV, dtype=F64)[:, None] * torch.sin(torch.deg2rad(th))[None, :]
    return torch.polar(torch.ones_like(ph), ph)


def _ula_grid(step):
    return -90.0 + step * torch.arange(grid_size(step), device=DEV, dtype=F64)


def _spectrum(B, a):
    """1 / |B^H a|^2 for factors B (..., M, K) and steering vectors a (M, L)."""
    out = []
    rows = max(1, int(2e8 // (B.shape[-1] * (B.shape[0] if B.dim() == 3 else 1) * 16)))
    for s in range(0, a.shape[1], rows):
        y = B.mH @ a[:, s:s + rows]
        out.append(1.0 / (y.real ** 2 + y.imag ** 2).sum(-2))
    return torch.cat(out, -1)


def _top(P, ok, d):
    """The d largest of the marked points of each row, in index order: (index, value), -1 / 0 where there are fewer."""
    v, i = torch.where(ok, P, -1.0).topk(d, dim=-1)
    n = P.shape[-1]
    i = torch.where(v > 0, i, n)
    i, at = i.sort(dim=-1)
    v = v.gather(-1, at)
    return torch.where(i < n, i, -1), torch.where(i < n, v, 0.0)


def _peaks(P, d):
    ok = torch.zeros_like(P, dtype=torch.bool)
    ok[..., 1:-1] = (P[..., 1:-1] > P[..., :-2]) & (P[..., 1:-1] > P[..., 2:])
    return _top(P, ok, d)


def _peaks2d(P, d, wrap):
    """P (B, Le, La): strictly larger than all neighbours, columns wrapping, rows outside absent."""
    B, Le, La = P.shape
    low = torch.full((B, Le + 2, La + 2), -1.0, dtype=P.dtype, device=DEV)
    low[:, 1:-1, 1:-1] = P
    if wrap:
        low[:, 1:-1, 0], low[:, 1:-1, -1] = P[:, :, -1], P[:, :, 0]
    ok = torch.ones_like(P, dtype=torch.bool)
    for r in range(3):
        for c in range(3):
            if (r, c) != (1, 1):
                ok &= P > low[:, r:r + Le, c:c + La]
    return _top(P.reshape(B, -1), ok.reshape(B, -1), d)


def _exact_chain(case, seed):
    X = _ula_snapshots(seed, 1, case["M"], case["N"], case["d"], 1.0 if case["M"] > 32 else 5.0, (0.0, 15.0))[0]
    R = _covariance(X)
    w, V = _subspace(R)
    P = _spectrum(_factor(w, V, case["d"], case["alg"]), _ula_steering(case["M"], _ula_grid(case["step"])))
    # the factor's columns are fixed only up to phases and rotations
    return {"R": R, "evals": w, "B": None, "P": P, "idx": None, "val": _peaks(P, case["d"])[1], "cnt": None}


def _algs(mask):
    return [a for a in range(4) if mask >> a & 1]


def _batch_parts(X, M, d, step, mask, per_chunk):
    """Chunks of (first, last, eigenvalues, eigenvectors, spectra (n, nalg, L))."""
    a = _ula_steering(M, _ula_grid(step))
    for s in range(0, X.shape[0], per_chunk):
        e = min(X.shape[0], s + per_chunk)
        w, V = _subspace(_covariance(X[s:e]))
        yield s, e, w, V, torch.stack([_spectrum(_factor(w, V, d, g), a) for g in _algs(mask)], 1)


def _exact_batch(case, seed):
    B, M, d, mask = case["B"], case["M"], case["d"], case["mask"]
    nalg, L = len(_algs(mask)), grid_size(case["step"])
    X = _ula_snapshots(seed, B, M, case["N"], d, 5.0, (0.0, 20.0))
    o = {"P": torch.zeros((B, nalg, L), dtype=F64, device=DEV), "evals": torch.zeros((B, M), dtype=F64, device=DEV),
         "val": torch.zeros((B, nalg, d), dtype=F64, device=DEV)}
    for s, e, w, V, P in _batch_parts(X, M, d, case["step"], mask, 128):
        o["P"][s:e], o["evals"][s:e], o["val"][s:e] = P, w, _peaks(P, d)[1]
    return {"status": None, **o, "idx": None, "cnt": None}


def _exact_uneven(case, seed):
    specs = _uneven_specs(case)
    buf, offs = _uneven_snapshots(case, seed, specs)
    steer = {}
    P, dmax = [], max(s[1] for s in specs)
    o = {"val": torch.zeros((len(specs), 1, dmax), dtype=F64, device=DEV), "evals": torch.zeros((len(specs), 64), dtype=F64, device=DEV)}
    for i, (M, d, N, step, alg) in enumerate(specs):
        if (M, step) not in steer:
            steer[M, step] = _ula_steering(M, _ula_grid(step))
        w, V = _subspace(_covariance(buf[int(offs[i]):int(offs[i]) + M * N].view(M, N)))
        p = _spectrum(_factor(w, V, d, alg), steer[M, step])
        o["val"][i, 0, :d], o["evals"][i, :M] = _peaks(p, d)[1], w
        P.append(p)
    return {"status": None, "P": torch.cat(P), "idx": None, "cnt": None, **o}


def _exact_circle_of(case, X, refine):
    M, La, Le, d, B = case["M"], case["La"], case["Le"], case["d"], X.shape[0]
    az = torch.deg2rad((2.0 if La == 180 else 1.0) * torch.arange(La, device=DEV, dtype=F64))
    el = torch.deg2rad((91 - Le) + torch.arange(Le, device=DEV, dtype=F64))
    u = torch.stack([torch.sin(el)[:, None] * torch.sin(az)[None], torch.sin(el)[:, None] * torch.cos(az)[None],
                     torch.cos(el)[:, None].expand(Le, La)]).reshape(3, -1)
    ph = 2.0 * math.pi * (torch.from_numpy(_circle_positions(M)).to(DEV) @ u)
    a = torch.polar(torch.ones_like(ph), ph)
    o = {"P": torch.zeros((B, Le, La), dtype=F64, device=DEV), "evals": torch.zeros((B, M), dtype=F64, device=DEV),
         "val": torch.zeros((B, 1, d), dtype=F64, device=DEV)}
    for s in range(0, B, 256):
        w, V = _subspace(_covariance(X[s:s + 256]))
        P = _spectrum(_factor(w, V, d, MUSIC), a).reshape(-1, Le, La)
        o["P"][s:s + 256], o["evals"][s:s + 256], o["val"][s:s + 256, 0] = P, w, _peaks2d(P, d, La == 360)[1]
    return {**o, "idx": None, "cnt": None, **({"angle": None} if refine else {})}


def _exact_circle(case, seed):
    return {"status": None, **_exact_circle_of(case, _circle_snapshots(seed, case["B"], case["M"], case["N"], case["d"]), case["refine"])}


def _refined(C, th, step):
    """The minimiser of a^H C a within a grid step of th (degrees), by bisection of its derivative; C (n, M, M), th (n, d)."""
    M = C.shape[-1]
    m = torch.arange(M, device=DEV, dtype=F64)
    lo, hi = torch.deg2rad(th - step), torch.deg2rad(th + step)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        ph = math.pi * m[None, :, None] * torch.sin(mid)[:, None, :]
        a = torch.polar(torch.ones_like(ph), ph)
        da = 1j * math.pi * m[None, :, None] * torch.cos(mid)[:, None, :] * a
        rising = ((da.conj() * (C @ a)).sum(1)).real > 0
        lo, hi = torch.where(rising, lo, mid), torch.where(rising, mid, hi)
    return torch.rad2deg(0.5 * (lo + hi))


def _roots(C, d):
    """Root form of one C (numpy, 64 bits): the d roots in the unit circle nearest to it, as ascending angles."""
    M = C.shape[0]
    r = np.roots([np.trace(C, offset=l) for l in range(M - 1, -M, -1)])
    r = r[np.abs(r) <= 1.0]
    r = r[np.argsort(-np.abs(r))[:d]]
    return np.sort(np.rad2deg(np.arcsin(np.clip(np.angle(r) / np.pi, -1.0, 1.0))))


def _exact_estimates(case, seed):
    B, M, d, step = case["B"], case["M"], case["d"], case["step"]
    X = _ula_snapshots(seed, B, M, case["N"], d, 8.0, (5.0, 20.0))
    L = grid_size(step)
    o = {"P": torch.zeros((B, 4, L), dtype=F64, device=DEV), "evals": torch.zeros((B, M), dtype=F64, device=DEV),
         "val": torch.zeros((B, 4, d), dtype=F64, device=DEV), "angle": torch.zeros((B, 4, d), dtype=F64, device=DEV),
         "root": torch.zeros((B, 4, d), dtype=F64, device=DEV)}
    for s, e, w, V, P in _batch_parts(X, M, d, step, 15, 256):
        at, val = _peaks(P, d)
        o["P"][s:e], o["evals"][s:e], o["val"][s:e] = P, w, val
        for g in range(4):
            Bf = _factor(w, V, d, g)
            C = Bf @ Bf.mH
            o["angle"][s:e, g] = torch.where(at[:, g] >= 0, _refined(C, -90.0 + step * at[:, g].to(F64), step), 0.0)
            host = C.cpu().numpy()
            o["root"][s:e, g] = torch.from_numpy(np.stack([_roots(c, d) for c in host])).to(DEV)
    cc = _estimate_circle(case)
    circle = _exact_circle_of(cc, _circle_snapshots(seed, case["circles"], cc["M"], cc["N"], cc["d"]), True)
    return {"status": None, "ula": {**o, "idx": None, "cnt": None, "order": None}, "circle": circle}


def _exact_svd(case, seed):
    X = _svd_snapshots(case, seed).to(C128)
    return {"evals": torch.linalg.svdvals(X) ** 2 / case["N"], "U": None}     # U up to a phase per column


def _exact_layers(net, x):
    """Activations of each layer (the last: logits) in 64 bits, from the network's 32-bit weights."""
    acts = [x.to(F64)]
    for l in range(4):
        z = acts[-1] @ net.buf["W"][l].to(F64).T + net.buf["b"][l].to(F64)
        acts.append(torch.relu(z) if l < 3 else z)
    return acts


def _exact_forward(case, seed):
    z = _exact_layers(_net(seed), _features(seed, case["B"]))[-1]
    return {"probs": torch.sigmoid(z), "logits": z}


def _exact_train(case, seed):
    net, B = _net(seed), case["B"]
    acts = _exact_layers(net, _features(seed, B))
    z, y = acts[-1], _labels(seed, B).to(F64)
    loss = (torch.clamp(z, min=0) - y * z + torch.log1p(torch.exp(-z.abs()))).sum() / B
    dz = (torch.sigmoid(z) - y) / B
    gW, gb = [None] * 4, [None] * 4
    for l in range(3, -1, -1):
        gW[l], gb[l] = dz.T @ acts[l], dz.sum(0)
        dz = (dz @ net.buf["W"][l].to(F64)) * (acts[l] > 0)
    b1, b2, eps, t = 0.9, 0.999, 1e-8, net.t + 1
    o = {"loss": loss.reshape(1), "gW": gW, "gb": gb, "W": [], "b": [], "mW": [], "mb": [], "vW": [], "vb": []}
    for l in range(4):
        for p, m, v, gr in (("W", "mW", "vW", gW[l]), ("b", "mb", "vb", gb[l])):
            mm = b1 * net.buf[m][l].to(F64) + (1 - b1) * gr
            vv = b2 * net.buf[v][l].to(F64) + (1 - b2) * gr * gr
            o[m].append(mm)
            o[v].append(vv)
            o[p].append(net.buf[p][l].to(F64) - 1e-4 * (mm / (1 - b1 ** t)) / (torch.sqrt(vv / (1 - b2 ** t)) + eps))
    return o


def _exact_windows(case, seed):
    B, d, w = case["B"], case["d"], case["width"]
    F, Pc, probs = _window_inputs(case, seed)
    m = torch.arange(16, device=DEV, dtype=F64)
    p, at = probs.clone(), torch.arange(B, device=DEV)
    o = torch.zeros((B, 8, w), dtype=F64, device=DEV)
    for k in range(min(d + 2, 8)):              # the highest bins, the neighbours of each pick suppressed
        bin_ = p.argmax(1)
        for off in (-1, 0, 1):
            p[at, (bin_ + off).clamp(0, 180)] = -1.0
        first = (bin_ * 1000 - w // 2).clamp(0, 180001 - w)
        for s in range(0, B, 128):
            th = torch.deg2rad(-90.0 + 0.001 * (first[s:s + 128, None] + torch.arange(w, device=DEV)[None]).to(F64))
            ph = math.pi * m[None, :, None] * torch.sin(th)[:, None, :]
            y = F[s:s + 128, :16 - d].conj() @ torch.polar(torch.ones_like(ph), ph)
            o[s:s + 128, k] = 1.0 / (y.real ** 2 + y.imag ** 2).sum(1)
    return {"spectra": o, "win": None, "idx": None, "val": None, "cnt": None, "fallback": None, "judge": None}


def exact(case, seed):
    f = {"chain": _exact_chain, "batch": _exact_batch, "uneven": _exact_uneven, "circle": _exact_circle,
         "estimates": _exact_estimates, "svd": _exact_svd, "forward": _exact_forward, "train": _exact_train, "windows": _exact_windows}[case["kind"]]
    return f(case, seed)
