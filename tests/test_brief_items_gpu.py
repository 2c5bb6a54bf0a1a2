"""The kernel for launches of many short streams: every output and state
against the oracle, at counts around steps and rows, requests that meet inside
rows, every step width, format and entry point, and on both sides of the rule
that chooses it."""
import os

import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 4


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _run(st, ops, states, ids, counts, fmt, entry="call", calls=2):
    """ops: the oracle's set of each stream, or one for all."""
    out = torch.empty(int(counts.sum()) + 8, dtype=torch.int32, device="cuda")
    plan = mtgp.mtgp_plan_create(st, ids, counts, fmt, out) if entry != "call" else None
    if entry == "traced plan":
        mtgp.mtgp_plan_set_trace(plan, True)
    for _ in range(calls):
        out.fill_(-1)
        if plan:
            mtgp.mtgp_plan_launch(plan)
        else:
            mtgp.mtgp_generate_f32(st, ids, counts, fmt, out)
        torch.cuda.synchronize()
        if isinstance(ops, list):
            ref = []
            for i, k in zip(ids, counts):
                o, states[i] = oracle.generate(ops[i], states[i], int(k), fmt)
                ref.append(o)
            ref = np.concatenate(ref)
        else:
            ref, states = oracle.generate_many(ops, states, ids, counts, fmt, THREADS)
        got = out.cpu().numpy().view(np.uint32)
        assert np.array_equal(got[:ref.size], ref)
        assert np.all(got[ref.size:] == 0xFFFFFFFF)
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
    mtgp.mtgp_check(st)
    if entry == "traced plan":
        t = mtgp.mtgp_plan_read_trace(plan)
        assert np.array_equal(np.sort(t[:, 3]), np.sort(counts)) and np.all(t[:, 1] >= t[:, 0])
    return mtgp.mtgp_plan_get_info(plan) if plan else None


def _edges(n, count):
    """`count` lengths around steps of 32, 64 and 128 and around rows of n."""
    e = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, n - 1, n, n + 1, 2 * n - 1, 2 * n, 2 * n + 1, 3 * n + 5, 4 * n]
    return np.array([e[i % len(e)] for i in range(count)], np.uint64)


@pytest.mark.parametrize("fmt", [0, 1, 2])
@pytest.mark.parametrize("mexp", [3217, 4253, 11213, 23209, 44497])
def test_counts_around_steps_and_rows(mexp, fmt):
    n = 8 * _sms() + 84
    p, op = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), oracle.params_generate(mexp, workloads.PARAM_SEED)
    seeds = np.arange(n, dtype=np.uint32)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    counts = _edges(mexp // 32 + 1, n)
    info = _run(mtgp.mtgp_init_statuses(p, seeds), op, states, seeds, counts, fmt, "plan" if fmt else "traced plan")
    assert info["resident_ctas_per_sm"] == 3 and info["config"]["warps_per_cta"] == 8   # the kernel in question


@pytest.mark.parametrize("cfg", [None, (2, 1, 4), (4, 4, 4), (8, 0, 8)])
def test_requests_that_meet_inside_rows(cfg):
    """Several requests per stream, claimed (more streams than warps) too."""
    n, rng = 8 * _sms() + 300, np.random.default_rng(5)
    p, op = mtgp.mtgp_params_generate(11213, 3), oracle.params_generate(11213, 3)
    seeds = np.arange(n, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses(p, seeds)
    if cfg:
        mtgp.mtgp_set_launch_config(st, warps_per_cta=cfg[0], ctas_per_sm=cfg[1], words_per_lane=cfg[2], kernel=0,
                                    coop_percent=0)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    ids = np.concatenate([seeds, rng.integers(0, n, 2 * n).astype(np.uint32)])
    counts = rng.choice([0, 1, 31, 100, 350, 351, 352], ids.size).astype(np.uint64)
    _run(st, op, states, ids, counts, 0)


@pytest.mark.parametrize("mexp,gap", [(11213, 255), (11213, 128), (11213, 127), (11213, 64), (23209, 128), (23209, 64),
                                      (3217, 64)])
def test_step_widths(mexp, gap):
    """pos = N - gap: steps of 128 words from 128 on, of 64 below."""
    n = 8 * _sms() + 50
    o0 = oracle.params_generate(mexp, 7)
    N = mexp // 32 + 1
    op = oracle.params_from_fields(mexp, N - gap, o0.sh1, o0.sh2, list(o0.rec_basis), list(o0.tmp_basis))
    p = mtgp.mtgp_params_create(mexp, N - gap, o0.sh1, o0.sh2, list(op.rec_tbl), list(op.tmp_tbl))
    seeds = np.arange(n, dtype=np.uint32)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    _run(mtgp.mtgp_init_statuses(p, seeds), op, states, seeds, _edges(N, n), 0)


def test_one_parameter_set_per_stream():
    n = 8 * _sms() + 20
    gs = [mtgp.mtgp_params_generate(11213, 40 + k) for k in range(5)]
    os_ = [oracle.params_generate(11213, 40 + k) for k in range(5)]
    seeds = np.arange(n, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses_multi(gs, seeds % 5, seeds)
    ops = [os_[s % 5] for s in range(n)]
    states = np.stack([oracle.init_state(ops[s], s) for s in range(n)])
    _run(st, ops, states, seeds, _edges(351, n), 2)


@pytest.mark.parametrize("over", ["no", "streams", "longest", "total"])
def test_both_sides_of_the_rule(over):
    sms, N = _sms(), 351
    n = 8 * sms + (0 if over == "streams" else 1)
    counts = np.full(n, 6 * N, np.uint64)
    counts[:4] = [8 * N, 1, 1, 1]
    counts[0] += over == "longest"
    if over == "total":
        counts[1:4] = 6 * N
    p, op = mtgp.mtgp_params_generate(11213, 3), oracle.params_generate(11213, 3)
    seeds = np.arange(n, dtype=np.uint32)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    info = _run(mtgp.mtgp_init_statuses(p, seeds), op, states, seeds, counts, 0, "plan")
    brief = info["resident_ctas_per_sm"] == 3 and info["config"]["warps_per_cta"] == 8
    assert brief == (over == "no")


@pytest.mark.parametrize("n_per_sm,rows", [(48, 12), (48, 13), (47, 8), (47, 9)])
def test_longest_stream_by_streams_per_sm(n_per_sm, rows):
    n = n_per_sm * _sms()
    counts = np.full(n, 40, np.uint64)
    counts[n // 3] = rows * 101
    p, op = mtgp.mtgp_params_generate(3217, 3), oracle.params_generate(3217, 3)
    seeds = np.arange(n, dtype=np.uint32)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    info = _run(mtgp.mtgp_init_statuses(p, seeds), op, states, seeds, counts, 0, "plan")
    brief = info["resident_ctas_per_sm"] == 3 and info["config"]["warps_per_cta"] == 8
    assert brief == (rows in (8, 12))
