"""The automatic launch shape of fused statistics: 16 warps per SM for even
streams, 8 for uneven ones; counts, outputs and states against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
GAP, HAM = (25, 5, 128), (25, 5, 1200, [585, 600, 615])


@pytest.mark.parametrize("mexp", [11213, 44497])
@pytest.mark.parametrize("even", [True, False])
def test_fused_automatic_shape(mexp, even):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 13 * sms + 5
    counts = np.full(n, 3 * (mexp // 32 + 1) + 5, np.uint64)
    if not even:
        counts[:9 * sms] //= 4   # the longest is a warp's share at 6 warps per SM
    p, op = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), oracle.params_generate(mexp, workloads.PARAM_SEED)
    seeds = np.arange(n, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses(p, seeds)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    out = torch.zeros(int(counts.sum()), dtype=torch.int32, device="cuda")
    plan = mtgp.mtgp_plan_create(st, seeds, counts, 0, out)
    mtgp.mtgp_plan_set_stats(plan, gap=GAP, hamming=HAM)
    assert mtgp.mtgp_plan_get_info(plan)["resident_ctas_per_sm"] == (2 if even else 1)
    mtgp.mtgp_plan_launch(plan)
    hist, table = mtgp.mtgp_plan_read_stats(plan)
    ref, states = oracle.generate_many(op, states, seeds, counts, 0, 4)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
    ends = np.cumsum(counts).astype(np.int64)
    for i in range(0, n, 7):
        x = ref[ends[i] - int(counts[i]):ends[i]]
        assert np.array_equal(hist[i], oracle.gap_histogram(x, *GAP))
        assert np.array_equal(table[i], oracle.hamming_pairs(x, *HAM))
