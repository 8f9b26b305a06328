"""The general-mode kernels at the edges of their work splits.

* the gather's residue blocks (B below, at and above 256, up to 4096) and its pairs per CTA (1, 2 or 4
  with the size of the call): bins against the oracle's FP64 HashToBins within 2e-5 of the hashing's
  largest bin (FP32 folds), and every request bit-identical to the same request run alone;
* the per-bin candidates and the selection of the k' largest: replayed by the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_1201_2501_gb300 import workloads
from tests.common import general_fields, oracle_params

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


def _plan(sf, f, batch, **over):
    p = sf.sfft_params_default(f["n"], f["k"], f["mode"])
    for name, _ in sf.SfftParams._fields_:
        if name in f:
            setattr(p, name, f[name])
    for name, v in over.items():
        setattr(p, name, v)
    return sf.Plan(p, batch)


def _signals(n, k, batch):
    return [workloads.general_noisy(n, k, workloads.seed_for(3, 300 + i)).x for i in range(batch)]


# (log2 n, k, batch): round 0 has B = 8 k; pairs per CTA 1, 2 and 4 from the call's pairs x residue blocks
@pytest.mark.parametrize("m,k,batch", [(10, 2, 1), (12, 32, 2), (12, 64, 1), (13, 128, 40), (12, 16, 100), (15, 512, 5)])
def test_gather_bins_match_oracle_at_every_split(sf, m, k, batch):
    n, seed = 1 << m, 91
    f = general_fields(n, k)
    P = oracle_params(f)
    xs = _signals(n, k, batch)
    plan = _plan(sf, f, batch)
    x = torch.as_tensor(np.stack(xs)).cuda()
    (idx, val, cnt, flag), tr = sf.sfft_execute_trace(plan, x, seed, f["z_cap"], 0)
    torch.cuda.synchronize()
    B = oracle.general_rounds(P)[1][0]
    _, _, dmax = oracle.locate_geometry(P, B)
    npairs = dmax * P.R_loc
    for s in {0, batch - 1}:
        bins = tr["bins"][s].cpu().numpy()
        bins = bins[..., 0] + 1j * bins[..., 1]
        rows = []
        for g in {0, 1, npairs - 1}:
            d = oracle.locate_draws(P, seed, s, 0, B, g // P.R_loc + 1, g % P.R_loc)
            rows += [(2 * g, d["sigma"], d["a"], d["b"]),
                     (2 * g + 1, d["sigma"], (d["a"] + d["beta"]) % n, d["b"])]
        for q in range(P.R_est):
            e = oracle.estimate_draws(P, seed, s, 0, q)
            rows.append((2 * npairs + q, e["sigma"], e["a"], e["b"]))
        for row, sg, aa, bb in rows:
            ob = oracle.hash_to_bins(xs[s].astype(np.complex128), sg, aa, bb, B, P.alpha0, P.delta)
            assert np.max(np.abs(bins[row] - ob)) <= 2e-5 * max(1.0, float(np.max(np.abs(ob)))), (s, row)
    for s in {0, batch // 2, batch - 1}:
        one = sf.sfft_execute_requests(plan, [x[s]], [seed], [s], f["z_cap"])
        torch.cuda.synchronize()
        c = int(cnt[s])
        assert int(one[2][0]) == c and int(one[3][0]) == int(flag[s])
        assert torch.equal(one[0][0, :c], idx[s, :c]) and torch.equal(one[1][0, :c], val[s, :c])
    plan.close()


# (log2 n, k, bins per k, batch): one, two and four bins per thread of the selection (B up to 1024, 2048,
# 4096), k' = 3 k above the sort's one key per thread (k = 512) and above B (every candidate is kept);
# zhat beyond the 2048 entries the finish takes at once, with many and with few bins (k = 1000)
@pytest.mark.parametrize("m,k,bpk,batch", [(12, 100, 8.0, 3), (13, 256, 8.0, 2), (14, 512, 8.0, 2), (12, 64, 2.0, 2),
                                           (8, 2, 8.0, 1), (14, 1000, 4.0, 2)])
def test_candidates_and_selection_match_oracle(sf, m, k, bpk, batch):
    """Every round replayed by the oracle on the pipeline's own bins: regions, bottoms and candidates
    bit for bit, the kept indices bit for bit, values within 1e-12 of the largest; the bins after the
    subtraction of zhat within 2e-5 of the hashing's largest bin before it (FP32 folds)."""
    n, seed = 1 << m, 17
    f = general_fields(n, k, bins_per_k=bpk, z_cap=min(4096, max(8 * k, 64)))
    P = oracle_params(f)
    xs = _signals(n, k, batch)
    x = torch.as_tensor(np.stack(xs)).cuda()
    plan = _plan(sf, f, batch)
    ks, Bs = oracle.general_rounds(P)
    for r in range(len(Bs)):
        _, tr = sf.sfft_execute_trace(plan, x, seed, f["z_cap"], r)
        torch.cuda.synchronize()
        tr = {key: v.cpu().numpy() for key, v in tr.items()}
        B = Bs[r]
        _, _, dmax = oracle.locate_geometry(P, B)
        npairs = dmax * P.R_loc
        for s in range(batch):
            bins = tr["bins"][s][..., 0] + 1j * tr["bins"][s][..., 1]
            d = [oracle.locate_draws(P, seed, s, r, B, D, q) for D in range(1, dmax + 1) for q in range(P.R_loc)]
            olfp, ovalid, ocand = oracle.locate_replay(P, B, d[0]["sigma"], d[0]["b"], [e["beta"] for e in d],
                                                       bins[0:2 * npairs:2], bins[1:2 * npairs:2])
            assert np.array_equal(tr["valid"][s], ovalid)
            assert np.array_equal(tr["regions"][s].view(np.uint64), olfp)
            want = np.where(ocand == oracle.BOTTOM, np.uint64(0xFFFFFFFF), ocand).astype(np.uint32)
            assert np.array_equal(tr["cand"][s].view(np.uint32), want)
            e = [oracle.estimate_draws(P, seed, s, r, q) for q in range(P.R_est)]
            wi, wv = oracle.estimate_from_bins(P, B, P.alpha0, [q["sigma"] for q in e], [q["b"] for q in e],
                                               [q["a"] for q in e], bins[2 * npairs:2 * npairs + P.R_est],
                                               np.unique(ocand[ocand != oracle.BOTTOM]), 3 * ks[r])
            nb, na = int(tr["zcount_before"][s]), int(tr["zcount_after"][s])
            zb, za = tr["zval_before"][s], tr["zval_after"][s]
            zi, zc = tr["zidx_before"][s][:nb].view(np.uint32).astype(np.uint64), zb[:nb, 0] + 1j * zb[:nb, 1]
            for row, h in [(0, (d[0]["sigma"], d[0]["a"], d[0]["b"])), (2 * npairs, (e[0]["sigma"], e[0]["a"], e[0]["b"])),
                           (2 * npairs - 1, (d[-1]["sigma"], (d[-1]["a"] + d[-1]["beta"]) % n, d[-1]["b"]))]:
                x64 = xs[s].astype(np.complex128)
                scale = np.max(np.abs(oracle.hash_to_bins(x64, *h, B, P.alpha0, P.delta)))
                assert np.max(np.abs(bins[row] - oracle.hash_to_bins(x64, *h, B, P.alpha0, P.delta, zi, zc))) <= 2e-5 * scale
            merged = dict(zip(tr["zidx_before"][s][:nb].view(np.uint32).tolist(), zb[:nb, 0] + 1j * zb[:nb, 1]))
            for i, v in zip(wi.astype(np.int64).tolist(), wv):
                merged[i] = merged[i] + v if i in merged else v
            keys = sorted(merged)[:f["z_cap"]]
            assert tr["zidx_after"][s][:na].view(np.uint32).tolist() == keys
            got, ref = za[:na, 0] + 1j * za[:na, 1], np.array([merged[i] for i in keys])
            assert np.max(np.abs(got - ref), initial=0.0) <= 1e-12 * max(1.0, float(np.max(np.abs(ref), initial=0.0)))
    plan.close()
