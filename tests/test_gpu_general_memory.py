"""General plans whose rounds take turns in the memory of one round: the same results, bit for bit."""
import numpy as np
import pytest

from paper_1201_2501_gb300 import workloads
from tests.common import general_fields

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("batch", [1, 2, 9])
def test_rounds_in_turn_equal_one_gather_for_all(batch):
    """n = 2^16, k = 16, alpha = 1/4: three rounds, two permuted copies.  A plan for 2 % of the device's memory
    in folds and copies beyond one round's gathers its rounds in turn, a plan for the batch alone at once."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2501_gb300 import build, sfft

    build.build()
    n, k = 1 << 16, 16
    f = general_fields(n, k, alpha0=0.25)
    p = sfft.sfft_params_default(n, k, sfft.SFFT_GENERAL)
    for name, _ in sfft.SfftParams._fields_:
        if name in f:
            setattr(p, name, f[name])
    extra = 900_000  # bytes per request
    many = torch.cuda.get_device_properties(0).total_memory // 50 // extra
    x = torch.as_tensor(np.stack([workloads.general_noisy(n, k, workloads.seed_for(3, 700 + i)).x
                                  for i in range(batch)])).cuda()
    got = []
    for max_batch in (batch, many):
        free = torch.cuda.mem_get_info()[0]
        plan = sfft.Plan(p, max_batch)
        if max_batch == many:  # one copy, not two
            assert (free - torch.cuda.mem_get_info()[0]) / many < 1_000_000
        for _ in range(2):
            out = [o.cpu().numpy() for o in sfft.sfft_execute(plan, x, 77, f["z_cap"])]
        torch.cuda.synchronize()
        got.append(out)
        plan.close()
    assert got[0][2].min() > 0
    for r in range(batch):
        c = got[0][2][r]
        assert got[1][2][r] == c and got[1][3][r] == got[0][3][r]
        assert np.array_equal(got[0][0][r, :c], got[1][0][r, :c])
        assert np.array_equal(got[0][1][r, :c], got[1][1][r, :c])
