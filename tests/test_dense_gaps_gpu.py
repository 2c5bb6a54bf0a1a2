"""Fused gap test with dense visits (one value in 2, 4 or 8): counts, outputs
and states against the oracle on both sides of the rule that resolves visits
by sub-step instead of by window."""
import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("b", [1, 2, 3, 4])
@pytest.mark.parametrize("mexp,split,fmt,ham", [
    (9689, 0, 0, (0, 8, 256, [120, 128, 136])), (11213, 0, 1, (25, 5, 1200, [585, 600, 615])),
    (11213, 700, 0, (0, 8, 512, [250, 260])), (23209, 0, 2, (0, 4, 128, [60, 64])), (44497, 3000, 0, None)])
def test_dense_visits(mexp, split, fmt, ham, b):
    N = mexp // 32 + 1
    counts = np.array([1, 31, N - 1, N, N + 1, 2 * N, 3 * N + 40, 9 * N + 1, 20 * N, 5000], np.uint64)
    n = counts.size
    p, op = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), oracle.params_generate(mexp, workloads.PARAM_SEED)
    ids = np.array([0, 1, 2, 3, 4, 5, 6, 7, 8, 3], np.uint32)   # two requests of one stream
    st = mtgp.mtgp_init_statuses(p, np.arange(n, dtype=np.uint32))
    states = np.stack([oracle.init_state(op, s) for s in range(n)])
    out = torch.zeros(int(counts.sum()), dtype=torch.int32, device="cuda")
    gap = (32 - b if fmt == 0 else 20, b, 40)
    plan = mtgp.mtgp_plan_create(st, ids, counts, fmt, out)
    mtgp.mtgp_plan_set_stats(plan, gap=gap, **({"hamming": ham} if ham else {}))
    if split:
        mtgp.mtgp_plan_set_split(plan, split)
    ends = np.cumsum(counts).astype(np.int64)
    for _ in range(2):
        mtgp.mtgp_plan_launch(plan)
        hist, table = mtgp.mtgp_plan_read_stats(plan)
        ref, states = oracle.generate_many(op, states, ids, counts, fmt, 4)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
        for i in range(n):
            x = ref[ends[i] - int(counts[i]):ends[i]]
            assert np.array_equal(hist[i], oracle.gap_histogram(x, *gap)), i
            if ham:
                assert np.array_equal(table[i], oracle.hamming_pairs(x, *ham)), i
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
