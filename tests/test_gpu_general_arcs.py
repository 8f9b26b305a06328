"""LocateInner's vote arcs of a whole turn and more."""
import numpy as np
import pytest

import oracle
from paper_1201_2501_gb300 import workloads
from tests.common import general_fields, oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("s", [0.999, 1.0, 1.0000001, 1.4999, 3.0])
@pytest.mark.parametrize("zero", [True, False])
def test_wide_arcs_decide_as_the_oracle(s, zero):
    """|beta theta - c| < s pi on the circle: for s = 1 only a vote exactly half a turn away misses, which the
    bins of a silent signal (c = 0) meet at most levels; beyond it none does.  Regions, bottom flags and
    candidates of every round are the oracle's on the same bins."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2501_gb300 import build, sfft

    build.build()
    n, k, batch, seed = 1 << 10, 8, 4, 99
    f = general_fields(n, k, s=s)
    P = oracle_params(f)
    p = sfft.sfft_params_default(n, k, sfft.SFFT_GENERAL)
    for name, _ in sfft.SfftParams._fields_:
        if name in f:
            setattr(p, name, f[name])
    plan = sfft.Plan(p, batch)
    x = np.stack([workloads.general_noisy(n, k, workloads.seed_for(3, 860 + i)).x for i in range(batch)])
    x = torch.as_tensor(x * (0.0 if zero else 1.0)).cuda()
    ks, Bs = oracle.general_rounds(P)
    for r, B in enumerate(Bs):
        _, tr = sfft.sfft_execute_trace(plan, x, seed, f["z_cap"], r)
        bins = tr["bins"].cpu().numpy()
        bins = bins[..., 0] + 1j * bins[..., 1]
        _, _, dmax = oracle.locate_geometry(P, B)
        npairs = dmax * P.R_loc
        for q in range(batch):
            d = [oracle.locate_draws(P, seed, q, r, B, D, i) for D in range(1, dmax + 1) for i in range(P.R_loc)]
            lfp, valid, cand = oracle.locate_replay(P, B, d[0]["sigma"], d[0]["b"], [e["beta"] for e in d],
                                                    bins[q, 0:2 * npairs:2], bins[q, 1:2 * npairs:2])
            assert np.array_equal(tr["valid"][q].cpu().numpy(), valid), (r, q)
            assert np.array_equal(tr["regions"][q].cpu().numpy().view(np.uint64), lfp), (r, q)
            want = np.where(cand == oracle.BOTTOM, np.uint64(0xFFFFFFFF), cand).astype(np.uint32)
            assert np.array_equal(tr["cand"][q].cpu().numpy().view(np.uint32), want), (r, q)
    plan.close()
