"""The late-tempering row loops (N - pos >= 256, and short states) and the per-SM claim lists:
every output and state against the oracle, tolerance zero, at the sizes where
they can go wrong: counts one off whole rows and whole passes of the unrolled
loop, requests that start and end inside rows, few items, and more items than
warps."""
import os

import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 4


def _check(mexp, ids, counts, fmt, n_streams, cfg=None, calls=2):
    p, op = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), oracle.params_generate(mexp, workloads.PARAM_SEED)
    seeds = np.arange(n_streams, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses(p, seeds)
    if cfg:
        mtgp.mtgp_set_launch_config(st, **cfg)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    ids, counts = np.asarray(ids, np.uint32), np.asarray(counts, np.uint64)
    for _ in range(calls):
        out = torch.full((int(counts.sum()) + 64,), -1, dtype=torch.int32, device="cuda")
        mtgp.mtgp_generate_f32(st, ids, counts, fmt, out)
        torch.cuda.synchronize()
        ref, states = oracle.generate_many(op, states, ids, counts, fmt, THREADS)
        got = out.cpu().numpy().view(np.uint32)
        assert np.array_equal(got[:ref.size], ref)
        assert np.all(got[ref.size:] == 0xFFFFFFFF)   # nothing behind the last request
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
    mtgp.mtgp_check(st)


@pytest.mark.parametrize("fmt", [0, 1, 2])
@pytest.mark.parametrize("mexp", [3217, 4253, 4423, 9689, 11213, 19937, 23209, 44497])
def test_counts_around_whole_rows(mexp, fmt):
    n = mexp // 32 + 1
    rows = [0, 1, 2, 3, 4, 5, 8, 9]
    counts = [max(r * n + d, 1) for r in rows for d in (-1, 0, 1, 31, 33)]
    _check(mexp, np.arange(len(counts)), counts, fmt, len(counts))


@pytest.mark.parametrize("mexp", [3217, 11213, 44497])
def test_requests_that_meet_inside_rows(mexp):
    n = mexp // 32 + 1
    rng = np.random.default_rng(mexp)
    ids = np.repeat(np.arange(20), 5)
    counts = rng.choice([1, 2, 31, n - 1, n, n + 1, 2 * n, 3 * n + 7, 700], ids.size)
    _check(mexp, ids, counts, 0, 20)


@pytest.mark.parametrize("n_items,cfg", [
    (1, None), (3, None), (151, None), (153, None), (607, None), (609, None), (1217, None), (2600, None),
    (2600, dict(warps_per_cta=4, ctas_per_sm=3, words_per_lane=4, coop_percent=0)),
    (2600, dict(warps_per_cta=2, ctas_per_sm=1, words_per_lane=4, coop_percent=0)),
    (700, dict(warps_per_cta=8, ctas_per_sm=1, words_per_lane=4, coop_percent=0))])
def test_every_item_is_claimed_once(n_items, cfg):
    counts = 352 + (np.arange(n_items) * 7919) % 1500
    _check(11213, np.arange(n_items), counts, 0, n_items, cfg, calls=1)
