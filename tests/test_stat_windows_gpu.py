"""The gap test's windows (32 ballots resolved at once) in the standalone
reduction and in the fused generation kernel, and the Hamming reduction's
look-ahead: counts against the oracle, at lengths around rounds, windows and
rows, for dense, sparse and missing visits."""
import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LENGTHS = [0, 1, 31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 2048, 16383, 16384, 16385, 17408, 33000]


@pytest.mark.parametrize("r,b,t", [(25, 5, 128), (0, 1, 7), (31, 1, 1023), (20, 12, 100), (0, 32, 1)])
@pytest.mark.parametrize("value", ["random", "all visits", "no visit"])
def test_gap_rounds(r, b, t, value):
    counts = np.array(LENGTHS, np.uint64)
    n = int(counts.sum())
    v = {"random": np.random.default_rng(b).integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32),
         "all visits": np.zeros(n, np.uint32), "no visit": np.full(n, 0xFFFFFFFF, np.uint32)}[value]
    got = mtgp.mtgp_gap_histogram(torch.from_numpy(v.view(np.int32)).cuda(), counts, r, b, t)
    ends = np.cumsum(counts).astype(np.int64)
    for i, e in enumerate(ends):
        assert np.array_equal(got[i], oracle.gap_histogram(v[e - int(counts[i]):e], r, b, t))


@pytest.mark.parametrize("r,s,L,bounds", [(25, 5, 1200, [585, 600, 615]), (0, 32, 64, [20, 30]), (0, 1, 40, []),
                                          (0, 32, 98304, [49000, 49152, 49300]), (10, 3, 768, [380])])
def test_hamming_pairs_ahead(r, s, L, bounds):
    counts = np.array(LENGTHS, np.uint64)
    v = np.random.default_rng(L).integers(0, 1 << 32, int(counts.sum()), dtype=np.uint64).astype(np.uint32)
    got = mtgp.mtgp_hamming_pairs(torch.from_numpy(v.view(np.int32)).cuda(), counts, r, s, L, bounds)
    ends = np.cumsum(counts).astype(np.int64)
    for i, e in enumerate(ends):
        assert np.array_equal(got[i], oracle.hamming_pairs(v[e - int(counts[i]):e], r, s, L, bounds))


# one row and two rows per window, a window that ends inside a row; Hamming
# per step (K >= 128) and per sub-step
@pytest.mark.parametrize("mexp", [3217, 9689, 11213, 19937, 44497])
@pytest.mark.parametrize("gap,ham", [((25, 5, 128), (25, 5, 1200, [585, 600, 615])), ((0, 1, 3), (0, 1, 40, [18, 22]))])
def test_fused_windows(mexp, gap, ham):
    n = mexp // 32 + 1
    counts = np.array([max(k * n + d, 1) for k in (0, 1, 2, 3, 4, 5) for d in (-1, 0, 1, 2)], np.uint64)
    p, op = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), oracle.params_generate(mexp, workloads.PARAM_SEED)
    seeds = np.arange(counts.size, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses(p, seeds)
    out = torch.zeros(int(counts.sum()), dtype=torch.int32, device="cuda")
    plan = mtgp.mtgp_plan_create(st, seeds, counts, 0, out)
    mtgp.mtgp_plan_set_stats(plan, gap=gap, hamming=ham)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    for _ in range(2):
        mtgp.mtgp_plan_launch(plan)
        hist, table = mtgp.mtgp_plan_read_stats(plan)
        ref, states = oracle.generate_many(op, states, seeds, counts, 0, 4)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
        ends = np.cumsum(counts).astype(np.int64)
        for i, e in enumerate(ends):
            x = ref[e - int(counts[i]):e]
            assert np.array_equal(hist[i], oracle.gap_histogram(x, *gap))
            assert np.array_equal(table[i], oracle.hamming_pairs(x, *ham))
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
