"""Exact-mode plans whose zhat may hold more than 256 entries (their rounds fold by residue blocks where B
is 512 or more, and decode with arrays sized by what was found) against the FP64 oracle, at the edges of
their ranges, and the same requests in a mixed batch.

Supports, counts and flags bit for bit; values within 1e-9 (FP64 data) or 1e-5 (FP32 data) of |X| = 1.
"""
import numpy as np
import pytest

import oracle
from paper_1201_2501_gb300 import workloads
from tests.common import exact_fields, oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def sf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2501_gb300 import build, sfft

    build.build()
    sfft.lib()
    return sfft


def _params(sf, f, prec):
    p = sf.sfft_params_default(f["n"], f["k"], f["mode"])
    for name, _ in sf.SfftParams._fields_:
        if name in f:
            setattr(p, name, f[name])
    p.precision = prec
    return p


# smallest such plan (z_cap 260); a capacity below k (CAPACITY, the smallest indices kept); FP64 at few
# samples; the longest ladder shifts (8 B, B = 1024); B = 4096; entries beyond shared memory (device
# memory in their place); chunks of 256 and of 8192 taps
@pytest.mark.parametrize("m,k,prec,batch,over", [
    (16, 65, 0, 3, {}), (16, 400, 1, 2, dict(z_cap=300)), (14, 100, 1, 2, dict(delta=1e-8)),
    (22, 130, 0, 2, dict(tau_dec=5e-3)), (18, 1000, 0, 2, {}),
    (20, 1500, 0, 1, dict(bins_per_k=2.5, z_cap=4096)), (16, 130, 0, 2, dict(chunk_taps=256)),
    (16, 130, 1, 2, dict(chunk_taps=8192))])
def test_large_plans_match_oracle(sf, m, k, prec, batch, over):
    n, seed = 1 << m, 33
    f = exact_fields(n, k, **{key: v for key, v in over.items() if key != "chunk_taps"})
    P = oracle_params(f)
    p = _params(sf, f, prec)
    p.chunk_taps = over.get("chunk_taps", 2048)
    dt = np.complex128 if prec else np.complex64
    sigs = [workloads.exact_sparse(n, k, workloads.seed_for(2, 700 + i), dtype=dt) for i in range(batch)]
    x = torch.as_tensor(np.stack([s.x for s in sigs])).cuda()
    plan, cap = sf.Plan(p, batch), f["z_cap"]
    small = sf.Plan(_params(sf, exact_fields(1 << 14, 8), prec), 1)
    idx, val, cnt, flag = [o.cpu().numpy() for o in sf.sfft_execute(plan, x, seed, cap)]
    bp = sf.BatchPlan([small, plan], batch + 1)
    xs = [x[r] for r in range(batch)]
    extra = torch.as_tensor(workloads.exact_sparse(1 << 14, 8, 5, dtype=dt).x).cuda()
    mixed = [o.cpu().numpy() for o in bp.execute([1] * batch + [0], xs + [extra], [seed] * (batch + 1),
                                                 list(range(batch)) + [0], cap)]
    for r, s in enumerate(sigs):
        oi, ov, of = oracle.sfft_exact(P, s.x.astype(np.complex128), seed, r)
        of = {0: sf.SFFT_OK, 1: sf.SFFT_ERR_NOT_CONVERGED, 2: sf.SFFT_ERR_CAPACITY}[of]
        c = int(cnt[r])
        assert np.array_equal(idx[r, :c].view(np.uint32).astype(np.int64), oi.astype(np.int64))
        assert int(flag[r]) == of
        assert np.max(np.abs(val[r, :c, 0] + 1j * val[r, :c, 1] - ov), initial=0.0) < (1e-9 if prec else 1e-5)
        assert int(mixed[2][r]) == c and int(mixed[3][r]) == of
        assert np.array_equal(mixed[0][r, :c], idx[r, :c]) and np.array_equal(mixed[1][r, :c], val[r, :c])
    for q in (bp, plan, small):
        q.close()


@pytest.mark.parametrize("m,k,t", [(14, 8, 0), (18, 64, 0), (22, 64, 1), (20, 128, 0)])
def test_fp64_decisions_at_their_boundaries(sf, m, k, t):
    """The FP64 data path takes a decision in FP32 only where FP64 agrees: bins whose magnitude, isolation,
    ladder rounding or re-estimation window lies 1e-12 to 1e-2 (relative) from its boundary, on both
    sides, decode as the oracle's FP64 does, bit for bit (values within 1e-12)."""
    n = 1 << m
    f = exact_fields(n, k)
    P = oracle_params(f)
    plan = sf.Plan(_params(sf, f, 1), 1)
    info = plan.round_info(t, seed=5)
    B, shifts = info["B"], info["shifts"]
    Np, L = n // B, len(shifts)
    rng = np.random.default_rng(m + t)
    near = lambda size: rng.choice([-1, 1], size) * 10.0 ** rng.uniform(-12, -2, size)
    for trial in range(24):
        sigma, b = int(rng.integers(0, n)) | 1, int(rng.integers(0, n))
        mag = np.where(rng.random(B) < 0.5, P.thr * (1 + near(B)), 10.0 ** rng.uniform(-0.5, 1, B))
        u = np.zeros((1 + L, B), dtype=np.complex128)
        u[0] = mag * np.exp(2j * np.pi * rng.random(B))
        c, M = np.zeros(B), 1.0
        for l in range(L - 1, -1, -1):  # coarsest first: th 2^logRatio - c / M close to a half-integer, or not
            ratio = Np / (shifts[l] // B) / M
            y = np.floor(rng.random(B) * ratio) + np.where(rng.random(B) < 0.5, 0.5 + near(B), 0.3 * rng.uniform(-1, 1, B))
            th = (y + c / M) / ratio
            c = c + M * (np.floor(y + 0.5) % ratio)
            M *= ratio
            size = np.where(rng.random(B) < 0.5, 1 + rng.choice([-1, 1], B) * P.iso_tol * (1 + near(B)), 1.0)
            u[l + 1] = u[0] * size * np.exp(-2j * np.pi * th)
        known = np.sort(rng.choice(n, size=max(2, B // 4), replace=False)).astype(np.uint32)
        for i in known:
            j, _ = oracle.bin_offset((sigma * (int(i) - b)) % n, n, B)
            edge = rng.choice([P.ref_lo, P.ref_hi]) * P.thr * (1 + float(near(1)[0]))
            for h, be in enumerate([0] + list(shifts)):
                u[h, j] = edge * np.exp(-2j * np.pi * ((be * sigma * int(i)) % n) / n)
        widx, wval, aux = sf.sfft_exact_decode(plan, t, sigma, b, torch.as_tensor(np.stack([u.real, u.imag], -1)).cuda(),
                                               torch.as_tensor(known.astype(np.int32)).cuda())
        torch.cuda.synchronize()
        cnt, nab, nkept = [int(v) for v in aux.cpu().numpy()]
        oi, ov, oab, okept = oracle.exact_decode(P, B, info["alpha"], sigma, b, shifts, u, known.astype(np.uint64),
                                                 with_kept=True)
        order = np.argsort(oi)
        assert (nab, nkept) == (oab, okept)
        assert np.array_equal(widx.cpu().numpy()[:cnt].astype(np.uint32).astype(np.int64), oi[order].astype(np.int64))
        v = wval.cpu().numpy()[:cnt]
        assert np.max(np.abs(v[:, 0] + 1j * v[:, 1] - ov[order]) / np.maximum(1.0, np.abs(ov[order])), initial=0.0) <= 1e-12
    plan.close()


@pytest.mark.parametrize("m,k,t", [(14, 8, 0), (18, 64, 0), (22, 64, 1)])
def test_fp64_decisions_on_magnitudes_below_fp32(sf, m, k, t):
    """The same where FP32 holds a magnitude or a product of two only as a denormal number or not at all:
    re-estimation windows at 1e-40 with residuals 1e-7 to 1e-3 (relative) from their ends, and ladder
    hashings of 1e-38 to 1 of u_0 under an isolation tolerance that lets them pass."""
    n = 1 << m
    f = exact_fields(n, k, thr=1e-8, ref_lo=1e-32, ref_hi=4e-32, iso_tol=2.0)
    P = oracle_params(f)
    plan = sf.Plan(_params(sf, f, 1), 1)
    info = plan.round_info(t, seed=5)
    B, shifts = info["B"], info["shifts"]
    Np, L = n // B, len(shifts)
    rng = np.random.default_rng(m + t)
    phases = lambda th: np.exp(-2j * np.pi * th)
    for trial in range(16):
        sigma, b = int(rng.integers(0, n)) | 1, int(rng.integers(0, n))
        u = np.zeros((1 + L, B), dtype=np.complex128)
        u[0] = 10.0 ** rng.uniform(-7.9, 0, B) * phases(rng.random(B))
        c, M = np.zeros(B), 1.0
        for l in range(L - 1, -1, -1):  # ladder roundings well away from a half-integer
            ratio = Np / (shifts[l] // B) / M
            y = np.floor(rng.random(B) * ratio) + 0.3 * rng.uniform(-1, 1, B)
            c, M, th = c + M * (np.floor(y + 0.5) % ratio), M * ratio, (y + c / M) / ratio
            u[l + 1] = u[0] * 10.0 ** rng.uniform(-38, 0, B) * phases(th)
        known = np.sort(rng.choice(n, size=max(2, B // 4), replace=False)).astype(np.uint32)
        for i in known:
            j, _ = oracle.bin_offset((sigma * (int(i) - b)) % n, n, B)
            off = float(rng.choice([-1, 1]) * 10.0 ** rng.uniform(-7, -3))
            edge = rng.choice([P.ref_lo, P.ref_hi]) * P.thr * (1 + off) * phases(rng.random())
            for h, be in enumerate([0] + list(shifts)):
                u[h, j] = edge * phases(((be * sigma * int(i)) % n) / n)
        widx, wval, aux = sf.sfft_exact_decode(plan, t, sigma, b, torch.as_tensor(np.stack([u.real, u.imag], -1)).cuda(),
                                               torch.as_tensor(known.astype(np.int32)).cuda())
        torch.cuda.synchronize()
        cnt, nab, nkept = [int(v) for v in aux.cpu().numpy()]
        oi, ov, oab, okept = oracle.exact_decode(P, B, info["alpha"], sigma, b, shifts, u, known.astype(np.uint64),
                                                 with_kept=True)
        order = np.argsort(oi)
        assert (nab, nkept, cnt) == (oab, okept, len(oi))
        assert np.array_equal(widx.cpu().numpy()[:cnt].astype(np.uint32).astype(np.int64), oi[order].astype(np.int64))
        v = wval.cpu().numpy()[:cnt]
        assert np.all(np.abs(v[:, 0] + 1j * v[:, 1] - ov[order]) <= 1e-12 * np.abs(ov[order]))
    plan.close()


@pytest.mark.parametrize("m,k", [(14, 8), (16, 130)])
def test_fp64_pruning_at_its_bound(sf, m, k):
    """|v| < prune thr is decided as FP64 decides it, also where FP32 cannot tell: with the bound a part in 1e9
    above (dropped) and below (kept) the magnitude of the smallest entry (3/4 of the others'), in a decode on
    chip and in one with arrays sized by what was found."""
    n, seed = 1 << m, 33
    f = exact_fields(n, k, delta=1e-8)
    dt = np.complex128
    s = workloads.exact_sparse(n, k, workloads.seed_for(2, 760), dtype=dt)
    X = np.zeros(n, dtype=dt)
    X[s.support] = s.values
    weak = int(s.support[k // 2])
    X[weak] *= 0.75
    x = torch.as_tensor(np.fft.ifft(X)[None]).cuda()

    def run(prune):
        plan = sf.Plan(_params(sf, dict(f, prune=prune), 1), 1)
        idx, val, cnt, flag = [o.cpu().numpy() for o in sf.sfft_execute(plan, x, seed, f["z_cap"])]
        plan.close()
        c = int(cnt[0])
        return idx[0, :c].view(np.uint32).astype(np.int64), val[0, :c, 0] + 1j * val[0, :c, 1]

    idx, val = run(f["prune"])
    assert np.array_equal(idx, s.support)
    size = float(np.abs(val[idx == weak])[0])
    kept, _ = run(size * (1 - 1e-9) / f["thr"])
    assert np.array_equal(kept, s.support)
    dropped, _ = run(size * (1 + 1e-9) / f["thr"])
    assert np.array_equal(dropped, s.support[s.support != weak])


@pytest.mark.parametrize("m,k", [(14, 8), (16, 130), (14, 100)])
def test_fp64_bins_at_the_threshold(sf, m, k):
    """Whole transforms with thr = 1 of coefficients of magnitude 1: the bins' magnitudes lie within the window's
    leakage (1e-8) of the threshold, on both sides, where FP32 cannot tell.  Supports, values and flags are the
    oracle's, in a decode on chip and in those with arrays sized by what was found."""
    n, seed, batch = 1 << m, 33, 3
    f = exact_fields(n, k, delta=1e-8, thr=1.0)
    P = oracle_params(f)
    sigs = [workloads.exact_sparse(n, k, workloads.seed_for(2, 770 + i), dtype=np.complex128) for i in range(batch)]
    plan = sf.Plan(_params(sf, f, 1), batch)
    idx, val, cnt, flag = [o.cpu().numpy() for o in sf.sfft_execute(
        plan, torch.as_tensor(np.stack([s.x for s in sigs])).cuda(), seed, f["z_cap"])]
    plan.close()
    missed = 0
    for r, s in enumerate(sigs):
        oi, ov, of = oracle.sfft_exact(P, s.x, seed, r)
        c = int(cnt[r])
        assert np.array_equal(idx[r, :c].view(np.uint32).astype(np.int64), oi.astype(np.int64))
        assert int(flag[r]) == {0: sf.SFFT_OK, 1: sf.SFFT_ERR_NOT_CONVERGED}[of]
        assert np.max(np.abs(val[r, :c, 0] + 1j * val[r, :c, 1] - ov), initial=0.0) < 1e-9
        missed += k - c
    assert 0 < missed < batch * k
