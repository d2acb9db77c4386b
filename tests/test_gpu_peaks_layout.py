"""Step-6 peak pickers (doa_peaks, doa_peaks2d) on spectra that start at every 4-byte offset from a
16-byte boundary, with plateaus and ties placed across the four-point groups the pickers load
together, rows shorter than four points, nearly flat rows, and d up to 63. Each case is compared
with the oracle's Step-6 on the same float32 values: indices and values bit-exact."""
import numpy as np
import pytest

import oracle
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return require_gpu()


def _view(torch, P, off):
    """A device view of P whose first element sits off floats past a 16-byte boundary."""
    buf = torch.zeros(P.size + 8, dtype=torch.float32, device="cuda")
    assert buf.data_ptr() % 16 == 0
    v = buf[off:off + P.size]
    v.copy_(torch.from_numpy(np.ascontiguousarray(P.reshape(-1), dtype=np.float32)))
    return v


def _peaks1d(torch, doa, P, off, d):
    v = _view(torch, P, off)
    idx = torch.full((max(d, 1),), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(max(d, 1), dtype=torch.float32, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    doa.doa_peaks(v, d, idx, val, cnt)
    torch.cuda.synchronize()
    n = cnt.item()
    return idx.cpu().numpy()[:n], val.cpu().numpy()[:n]


def _peaks2d(torch, doa, P, off, wrap, d):
    Le, La = P.shape
    v = _view(torch, P, off)
    idx = torch.full((max(d, 1),), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(max(d, 1), dtype=torch.float32, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    doa.doa_peaks2d(v, La, Le, wrap, d, idx, val, cnt)
    torch.cuda.synchronize()
    n = cnt.item()
    return idx.cpu().numpy()[:n], val.cpu().numpy()[:n]


def _plateaus(rng, L):
    """Integer levels with runs of equal values that start and end at every position mod 4."""
    P = rng.integers(0, 6, L).astype(np.float32)
    for start in range(1, max(L - 8, 1), 7):
        n = 1 + (start % 6)
        P[start:start + n] = 9.0 + (start % 3)
    return P


@pytest.mark.parametrize("L", [3, 4, 5, 6, 7, 8, 9, 31, 1023, 1024, 1025, 4097, 18001])
def test_peaks_every_offset(env, L):
    torch, doa = env
    rng = np.random.default_rng(L)
    spectra = [_plateaus(rng, L), rng.random(L).astype(np.float32)]
    x = np.linspace(0.0, 9.0, L)
    spectra.append((np.cos(x) ** 2 + 1e-3 * np.cos(37 * x)).astype(np.float32))   # smooth, few peaks
    for P in spectra:
        for off in range(4):
            for d in (1, 4, 63):
                gi, gv = _peaks1d(torch, doa, P, off, d)
                ri, rv = oracle.peaks(P.astype(np.float64), d)
                assert gi.tolist() == ri.tolist(), (L, off, d)
                assert np.array_equal(gv.astype(np.float64), rv), (L, off, d)


def test_peaks_many_selections(env):
    """d = 63 on noise: the winning threads' four-entry caches run dry and are refilled many times
    inside the warp rounds."""
    torch, doa = env
    rng = np.random.default_rng(63)
    for L in (18001, 360001):
        P = rng.random(L).astype(np.float32)
        P[::97] = 2.0 + rng.integers(0, 3, P[::97].size)          # many equal tall peaks
        for off in range(4):
            gi, gv = _peaks1d(torch, doa, P, off, 63)
            ri, rv = oracle.peaks(P.astype(np.float64), 63)
            assert len(ri) == 63
            assert gi.tolist() == ri.tolist(), (L, off)
            assert np.array_equal(gv.astype(np.float64), rv)


@pytest.mark.parametrize("Le,La", [(5, 1), (3, 2), (7, 3), (4, 4), (3, 5), (2, 6), (9, 7), (6, 13), (90, 360),
                                   (5, 361)])
def test_peaks2d_every_offset(env, Le, La):
    torch, doa = env
    rng = np.random.default_rng(Le * 1000 + La)
    spectra = [rng.integers(0, 4, (Le, La)).astype(np.float32), rng.random((Le, La)).astype(np.float32)]
    # rows that are nearly flat along the azimuth (as near the pole of a circular array), then a lobe
    a = np.arange(La)[None, :]
    e = np.arange(Le)[:, None]
    lobe = np.cos(2 * np.pi * a / max(La, 1)) * np.exp(-0.1 * e) + 0.05 * e
    jitter = rng.integers(0, 3, (Le, La)) * 1e-6
    spectra.append((lobe * (e > Le // 3) + 1.0 + jitter).astype(np.float32))
    for P in spectra:
        for wrap in (False, True):
            for off in range(4):
                for d in (1, 5, 63):
                    gi, gv = _peaks2d(torch, doa, P, off, wrap, d)
                    ri, rv = oracle.peaks2d(P.astype(np.float64), d, wrap)
                    assert gi.tolist() == ri.tolist(), (Le, La, wrap, off, d)
                    assert np.array_equal(gv.astype(np.float64), rv), (Le, La, wrap, off, d)


@pytest.mark.parametrize("L,off,d", [(16383, 0, 5), (16384, 1, 7), (16389, 3, 63), (40003, 2, 1), (360001, 0, 8)])
def test_peaks_cluster_matches_oracle(env, L, off, d):
    """Spectra on both sides of the length from which a cluster of CTAs searches one, at several alignment
    offsets, with plateaus: bit-exact indices and values, alone and in a batch of few long spectra."""
    torch, doa = env
    rng = np.random.default_rng(L + d)
    P = rng.integers(1, 40 if d > 20 else 4000, size=L).astype(np.float32)      # ties and plateaus
    buf = torch.zeros(L + off, dtype=torch.float32, device="cuda")
    buf[off:].copy_(torch.from_numpy(P))
    idx = torch.full((d,), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(d, dtype=torch.float32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    doa.doa_peaks(buf[off:], d, idx, val, cnt, L=L)
    torch.cuda.synchronize()
    oi, ov = oracle.peaks(P.astype(np.float64), d)
    n = int(cnt.item())
    assert list(idx.cpu().numpy()[:n]) == list(oi)
    assert np.array_equal(val.cpu().numpy()[:n].astype(np.float64), ov)
    if L % 2 == 1 and L >= 16384:      # the 2-D rule on the same points as one wrapped row
        i2 = torch.full((d,), -1, dtype=torch.int32, device="cuda")
        doa.doa_peaks2d(buf[off:], L, 1, True, d, i2, val, cnt)
        torch.cuda.synchronize()
        w = (P > np.roll(P, 1)) & (P > np.roll(P, -1))
        k = np.nonzero(w)[0]
        k = np.sort(k[np.lexsort((k, -P[k]))][:d])
        assert list(i2.cpu().numpy()[:int(cnt.item())]) == list(k)


@pytest.mark.parametrize("L,d", [(181, 1), (1801, 3), (1023, 0)])
def test_many_spectra_match_the_single_picker(env, L, d):
    """A batch of enough spectra takes a small CTA for each: the picks are those of doa_peaks on the
    spectra the same solve wrote (3200 jobs, spectra starting at odd offsets)."""
    torch, doa = env
    B, M, N, mask = 800, 4, 64, 0xF
    gen = torch.Generator(device="cuda").manual_seed(L)
    X = torch.view_as_complex(torch.randn(B, M, N, 2, generator=gen, device="cuda"))
    P = torch.zeros(B * 4 * L + 1, device="cuda")[1:].view(B, 4 * L)
    dk = max(d, 1)
    idx = torch.full((B, 4 * dk), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros((B, 4 * dk), device="cuda")
    cnt = torch.full((B, 4), -1, dtype=torch.int32, device="cuda")
    probs = [doa.make_problem(X[i], d, mask, doa.grid(-90.0, 180.0 / (L - 1), L), P[i], idx[i] if d else None,
                              val[i] if d else None, cnt[i], None) for i in range(B)]
    plan = doa.BatchPlan(probs)
    status = torch.full((B,), -1, dtype=torch.int32, device="cuda")
    doa.doa_solve_batch(plan, doa.workspace(plan), status)
    torch.cuda.synchronize()
    assert int(status.abs().max()) == 0
    for i in range(0, B, 37):
        for a in range(4):
            i1 = torch.full((dk,), -1, dtype=torch.int32, device="cuda")
            v1 = torch.zeros(dk, device="cuda")
            c1 = torch.zeros(1, dtype=torch.int32, device="cuda")
            doa.doa_peaks(P[i, a * L:(a + 1) * L], d, i1, v1, c1)
            n = int(c1)
            assert int(cnt[i, a]) == n
            assert torch.equal(idx[i, a * d:a * d + n], i1[:n]) and torch.equal(val[i, a * d:a * d + n], v1[:n])


@pytest.mark.parametrize("L,off,d", [(4095, 1, 5), (4096, 0, 9), (4101, 3, 63), (8191, 2, 1)])
def test_peaks_around_the_shortest_cluster(env, L, off, d):
    test_peaks_cluster_matches_oracle(env, L, off, d)


def test_peaks_of_the_longest_spectra(env):
    """2^31 - 64 points, where an index four quads ahead of a spectrum's last ones is beyond an int: peaks at
    both ends and around the last steps, found exactly."""
    torch, doa = env
    L = 2 ** 31 - 64
    free, _ = torch.cuda.mem_get_info()
    if free < 6 * L:
        pytest.skip("needs 12 GB")
    P = torch.zeros(L, dtype=torch.float32, device="cuda")
    at = [1, 4097, L // 2 + 3, L - 70001, L - 24581, L - 24577, L - 8190, L - 5, L - 2]
    for k, i in enumerate(at):
        P[i] = float(k + 1)
    idx = torch.full((16,), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(16, dtype=torch.float32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    doa.doa_peaks(P, 16, idx, val, cnt)
    torch.cuda.synchronize()
    assert cnt.item() == len(at)
    assert idx.cpu().tolist()[:len(at)] == at
    assert val.cpu().tolist()[:len(at)] == [float(k + 1) for k in range(len(at))]
