"""The general-mode kernels at the edges of their work splits.

* the gather's residue blocks (B below, at and above 256, up to 4096) and its pairs per CTA (1, 2 or 4
  with the size of the call): bins against the oracle's FP64 HashToBins within 2e-5 of the hashing's
  largest bin (FP32 folds), and every request bit-identical to the same request run alone.
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
