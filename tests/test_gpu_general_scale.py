"""LocateSignal's decisions do not depend on the scale of the signal, as far as FP32 samples reach."""
import numpy as np
import pytest

import oracle
from paper_1201_2501_gb300 import workloads
from tests.common import general_fields, oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,k", [(12, 4), (14, 40)])
@pytest.mark.parametrize("scale", [-80, -64, 63, 70])
def test_regions_and_candidates_of_a_scaled_signal(m, k, scale):
    """A signal times a power of two has the bins times that power, in FP32 too: the same regions, bottom flags
    and candidates in every round, and the values times the power (to 1e-6: samples of 2^-80 under window taps
    of 1e-6 reach the denormal numbers)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2501_gb300 import build, sfft

    build.build()
    n, batch, seed = 1 << m, 3, 606
    f = general_fields(n, k)
    p = sfft.sfft_params_default(n, k, sfft.SFFT_GENERAL)
    for name, _ in sfft.SfftParams._fields_:
        if name in f:
            setattr(p, name, f[name])
    plan = sfft.Plan(p, batch)
    x = torch.as_tensor(np.stack([workloads.general_noisy(n, k, workloads.seed_for(3, 820 + i)).x
                                  for i in range(batch)])).cuda()
    for r in range(len(oracle.general_rounds(oracle_params(f))[0])):
        (out0, tr0), (out1, tr1) = (sfft.sfft_execute_trace(plan, x * s, seed, f["z_cap"], r) for s in (1.0, 2.0 ** scale))
        for name in ("valid", "regions", "cand"):
            assert torch.equal(tr0[name], tr1[name]), (r, name)
        assert bool(tr0["valid"].any())
        for s in range(batch):
            c = int(out0[2][s])
            assert int(out1[2][s]) == c > 0 and torch.equal(out0[0][s, :c], out1[0][s, :c])
            want = out0[1][s, :c]
            assert float((out1[1][s, :c] * 2.0 ** -scale - want).abs().max()) <= 1e-6 * float(want.abs().max())
    plan.close()
