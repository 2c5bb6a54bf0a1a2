"""The work that users of this library have it do, as measurable cases.

Every case goes through the public Python binding (paper_1501_07701_gb300.mtgp)
as a program of a user does.  A case is a dict of plain values; its "do" names
the entry point:

  call   mtgp_generate_u32 / _f32 on resident streams (work table per call)
  plan   mtgp_plan_launch of a recorded plan (unsplit or split, tuned or not)
  stats  mtgp_plan_launch of a plan with fused statistics, then
         mtgp_plan_read_stats
  mt     mtgp_mt_generate, the comparison generator
  jump   mtgp_jump of many streams, then a draw from each of them
  tests  mtgp_gap_histogram and mtgp_hamming_pairs over numbers in memory
  serve  a burst of requests through mtgp_server_submit / _progress

Sizes are those of paper_1501_07701_gb300/workloads.py, README.md, bench.py
and the tests.  Parameter sets are seed-generated from workloads.PARAM_SEED;
the streams' seed statuses, and so all numbers, come from the seed given to
prepare().
"""
import math

import numpy as np
import torch

from paper_1501_07701_gb300 import mtgp, quality, workloads

FORMATS = {"u32": mtgp.MTGP_U32, "f32_12": mtgp.MTGP_F32_12, "f32_01": mtgp.MTGP_F32_01}
HAMMING = (25, 5, 1200)          # r, s, L of test 100
GAP = (25, 5, 128)               # r, b, t of test 35


def listed():
    return [
        # A running simulation asks one of its resident streams for the
        # smallest request of the serving workload: latency and launches.
        {"name": "call-1x256", "do": "call", "mexp": 11213, "streams": 1, "resident": 4096,
         "lo": 8.0, "hi": 8.0, "fmt": "u32", "sets": 0},
        # README quick start: 4096 streams, 1000 numbers each, one direct call.
        {"name": "call-4096x1000", "do": "call", "mexp": 11213, "streams": 4096, "resident": 4096,
         "lo": math.log2(1000), "hi": math.log2(1000), "fmt": "u32", "sets": 0},
        # One long stream (the "single" workload, 2^20 numbers), shared out
        # over 64 pieces that start from exact jumps.
        {"name": "plan-1x2^20-split", "do": "plan", "mexp": 11213, "streams": 1, "lo": 20.0, "hi": 20.0,
         "fmt": "u32", "sets": 0, "split": 16384, "tune": True},
        # The "equal" workload as a plan that its user did not tune.
        {"name": "plan-4096x2^18", "do": "plan", "mexp": 11213, "streams": 4096, "lo": 18.0, "hi": 18.0,
         "fmt": "u32", "sets": 0, "split": 0, "tune": False},
        # The "long" workload at the largest exponent, as floats in [1, 2).
        {"name": "plan-1024x2^20-44497", "do": "plan", "mexp": 44497, "streams": 1024, "lo": 20.0,
         "hi": 20.0, "fmt": "f32_12", "sets": 0, "split": 0, "tune": True},
        # The headline: the "uneven" workload, 10 000 streams of 2^10 .. 2^22
        # numbers, tuned.
        {"name": "plan-uneven", "do": "plan", "mexp": 11213, "streams": 10000, "lo": 10.0, "hi": 22.0,
         "fmt": "u32", "sets": 0, "split": 0, "tune": True},
        # The same at the paper's own exponent, long streams split.
        {"name": "plan-uneven-3217-split", "do": "plan", "mexp": 3217, "streams": 10000, "lo": 10.0,
         "hi": 22.0, "fmt": "u32", "sets": 0, "split": 701932, "tune": True},
        # The uneven workload with tests 35 and 100 counted while it is
        # generated, in the split shape that the benchmark reports.
        {"name": "stats-uneven-split", "do": "stats", "mexp": 11213, "streams": 10000, "lo": 10.0,
         "hi": 22.0, "fmt": "u32", "sets": 0, "split": 1052897, "tune": False},
        # The comparison generator at the paper's exponent, uneven workload.
        {"name": "mt-uneven-3217", "do": "mt", "p": 3217, "streams": 10000, "lo": 10.0, "hi": 22.0,
         "fmt": "u32"},
        # Spacing 10 000 streams 2^40 numbers apart, then a first draw of each.
        {"name": "jump-10000", "do": "jump", "mexp": 11213, "streams": 10000, "jump": 1 << 40, "draw": 64},
        # Both tests over the equal workload's numbers already in memory.
        {"name": "tests-4096x2^18", "do": "tests", "streams": 4096, "lo": 18.0, "hi": 18.0},
        # A burst of requests of the serving workload (2^8 .. 2^20 numbers,
        # u32 or f32 in [0, 1)) over 65 536 resident streams, long ones split.
        {"name": "serve-burst-48", "do": "serve", "mexp": 11213, "resident": 65536, "requests": 48,
         "lo": 8.0, "hi": 20.0, "max_piece": 65536},
    ]


def _log_int(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))


def draw(rng):
    """One more case of the same ranges (at most 2^31 numbers)."""
    do = rng.choice(["call", "call", "plan", "plan", "plan", "stats", "mt", "jump", "tests", "serve"])
    c = {"do": do}
    if do in ("call", "plan", "stats"):
        c["mexp"] = rng.choice([3217, 11213, 11213, 23209, 44497])
    if do in ("call", "plan", "mt", "stats"):
        c["fmt"] = rng.choice(["u32", "f32_12", "f32_01"])
    if do in ("call", "plan"):
        c["sets"] = rng.choice([0, 0, 0, 7])
    if do == "call":
        c["streams"] = _log_int(rng, 1, 4096)
        c["resident"] = max(c["streams"], _log_int(rng, 64, 8192))
        c["lo"] = rng.uniform(5.0, 12.0)
        c["hi"] = c["lo"] + rng.choice([0.0, 3.0, 6.0])
    elif do == "plan":
        c["streams"] = _log_int(rng, 1, 10000)
        top = min(22.0, 31.0 - math.log2(c["streams"]))
        c["hi"] = rng.uniform(12.0, top)
        c["lo"] = c["hi"] - rng.choice([0.0, 0.0, 6.0, 10.0])
        c["split"] = rng.choice([0, 0, 16384, 262144]) if c["mexp"] in (3217, 11213) and not c["sets"] else 0
        c["tune"] = rng.choice([True, False])
    elif do == "stats":
        c["sets"] = 0
        c["streams"] = _log_int(rng, 64, 10000)
        c["hi"] = min(21.0, 30.0 - math.log2(c["streams"])) - rng.uniform(0.0, 3.0)
        c["lo"] = c["hi"] - rng.choice([0.0, 6.0])
        c["split"] = rng.choice([0, 262144]) if c["mexp"] in (3217, 11213) else 0
        c["tune"] = False
    elif do == "mt":
        c["p"] = rng.choice([3217, 3217, 19937])
        c["streams"] = _log_int(rng, 1, 10000)
        top = min(22.0, 31.0 - math.log2(c["streams"]))
        c["hi"] = rng.uniform(10.0, top)
        c["lo"] = c["hi"] - rng.choice([0.0, 5.0, 9.0])
    elif do == "jump":
        c["mexp"] = rng.choice([3217, 11213, 23209])
        c["streams"] = _log_int(rng, 1, 10000 if c["mexp"] < 20000 else 2000)
        c["jump"] = _log_int(rng, 1 << 16, 1 << 50)
        c["draw"] = _log_int(rng, 16, 1024)
    elif do == "tests":
        c["streams"] = _log_int(rng, 1, 10000)
        top = min(22.0, 30.0 - math.log2(c["streams"]))
        c["hi"] = rng.uniform(10.0, top)
        c["lo"] = c["hi"] - rng.choice([0.0, 0.0, 6.0])
    else:
        c["mexp"] = rng.choice([3217, 11213, 23209])
        c["resident"] = _log_int(rng, 256, 65536)
        c["requests"] = rng.randint(8, 60)
        c["lo"] = 8.0
        c["hi"] = rng.uniform(10.0, 20.0)
        c["max_piece"] = rng.choice([0, 65536]) if c["mexp"] < 20000 else 0
    return c


def _counts(case):
    """Numbers per request: equal, or the uneven workload's log-uniform draw."""
    n = case.get("streams") or case["requests"]
    if case["lo"] == case["hi"]:
        return np.full(n, int(round(2.0 ** case["hi"])), np.uint64)
    return workloads.uneven_counts(n, case["lo"], case["hi"], seed=7)


def _ids(case, seed):
    """Streams that a call or burst touches: some of the resident ones."""
    n = case.get("streams") or case["requests"]
    if n > case["resident"] // 2:
        return np.arange(n, dtype=np.uint32) % case["resident"]
    return np.random.default_rng(seed).choice(case["resident"], n, replace=False).astype(np.uint32)


def _seeds(n, seed):
    return (np.arange(n, dtype=np.uint64) + np.uint64(seed) * np.uint64(1000003)).astype(np.uint32)


def _streams(case, n, seed):
    sets = case.get("sets", 0)
    if not sets:
        return mtgp.mtgp_init_statuses(mtgp.mtgp_params_generate(case["mexp"], workloads.PARAM_SEED),
                                       _seeds(n, seed))
    ps = workloads.param_seeds(n, sets)[:sets]
    return mtgp.mtgp_init_statuses_multi([mtgp.mtgp_params_generate(case["mexp"], int(s)) for s in ps],
                                         np.arange(n) % len(ps), _seeds(n, seed))


def _buffer(case, total):
    return torch.empty(total, dtype=torch.int32 if case["fmt"] == "u32" else torch.float32, device="cuda")


class _Arena:
    """The server's device arena, as torch takes device memory of others.
    torch keeps this object while a tensor views the memory, and it keeps the
    server, which owns the memory."""

    def __init__(self, server, words):
        self.server = server
        self.__cuda_array_interface__ = {"shape": (words,), "typestr": "<i4", "version": 3,
                                         "data": (mtgp.mtgp_server_arena(server), False)}


def prepare(case, seed):
    do = case["do"]
    s = {"case": case, "do": do}
    if do == "call":
        s["streams"] = _streams(case, case["resident"], seed)
        s["ids"], s["counts"] = _ids(case, seed), _counts(case)
        s["out"] = _buffer(case, int(s["counts"].sum()))
    elif do in ("plan", "stats"):
        n = case["streams"]
        s["counts"] = _counts(case)
        s["out"] = _buffer(case, int(s["counts"].sum()))
        s["streams"] = _streams(case, n, seed)
        if do == "stats":
            mtgp.mtgp_set_launch_config(s["streams"], **dict(mtgp.mtgp_get_launch_config(s["streams"]),
                                                             warps_per_cta=8, ctas_per_sm=2))
        s["plan"] = mtgp.mtgp_plan_create(s["streams"], np.arange(n), s["counts"], FORMATS[case["fmt"]],
                                          s["out"])
        if do == "stats":
            mtgp.mtgp_plan_set_stats(s["plan"], gap=GAP,
                                     hamming=HAMMING + (quality.default_hamming_bounds(1200, 4),))
        if case["split"]:
            mtgp.mtgp_plan_set_split(s["plan"], case["split"])
        if case["tune"]:
            mtgp.mtgp_plan_autotune(s["plan"])
    elif do == "mt":
        n = case["streams"]
        q = mtgp.mtgp_mt_params_mt19937() if case["p"] == 19937 else \
            mtgp.mtgp_mt_params_generate(case["p"], workloads.PARAM_SEED)
        s["mt"] = mtgp.mtgp_mt_init(q, _seeds(n, seed))
        s["ids"], s["counts"] = np.arange(n, dtype=np.uint32), _counts(case)
        s["out"] = _buffer(case, int(s["counts"].sum()))
    elif do == "jump":
        n = case["streams"]
        s["streams"] = _streams(case, n, seed)
        s["ids"] = np.arange(n, dtype=np.uint32)
        s["jumps"] = np.full(n, case["jump"], np.uint64)
        s["counts"] = np.full(n, case["draw"], np.uint64)
        s["out"] = torch.empty(n * case["draw"], dtype=torch.int32, device="cuda")
    elif do == "tests":
        s["counts"] = _counts(case)
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        s["values"] = torch.randint(-(1 << 31), 1 << 31, (int(s["counts"].sum()),), dtype=torch.int32,
                                    device="cuda", generator=g)
        s["bounds"] = quality.default_hamming_bounds(1200, 4)
    else:
        s["streams"] = _streams(case, case["resident"], seed)
        s["server"] = mtgp.mtgp_server_create(s["streams"], arena_bytes=1 << 30, max_piece=case["max_piece"])
        s["arena"] = torch.as_tensor(_Arena(s["server"], (1 << 30) // 4), device="cuda")
        s["held"] = []
        s["ids"], s["counts"] = _ids(case, seed), _counts(case)
    return s


def _serve(s):
    server, done = s["server"], {}
    for c in s["held"]:   # the last burst's results have been used
        mtgp.mtgp_server_release(server, c["arena_offset"], c["count"])
    for j, (i, k) in enumerate(zip(s["ids"].tolist(), s["counts"].tolist())):
        mtgp.mtgp_server_submit(server, i, k, mtgp.MTGP_F32_01 if j % 2 else mtgp.MTGP_U32, j)
    while len(done) < len(s["ids"]):
        for c in mtgp.mtgp_server_progress(server, 64):
            done[c["tag"]] = c
    out = []
    for j in range(len(done)):
        c = done[j]
        v = s["arena"][c["arena_offset"]:c["arena_offset"] + c["count"]]
        out.append(v.view(torch.float32) if c["fmt"] == mtgp.MTGP_F32_01 else v)
    s["held"] = list(done.values())
    return out


def run(state):
    s, do = state, state["do"]
    if do == "call":
        if s["case"]["fmt"] == "u32":
            mtgp.mtgp_generate_u32(s["streams"], s["ids"], s["counts"], s["out"])
        else:
            mtgp.mtgp_generate_f32(s["streams"], s["ids"], s["counts"], FORMATS[s["case"]["fmt"]], s["out"])
        return s["out"]
    if do == "plan":
        mtgp.mtgp_plan_launch(s["plan"])
        return s["out"]
    if do == "stats":
        mtgp.mtgp_plan_launch(s["plan"])
        hist, table = mtgp.mtgp_plan_read_stats(s["plan"])
        return [s["out"], hist.view(np.int64), table.view(np.int64)]
    if do == "mt":
        mtgp.mtgp_mt_generate(s["mt"], s["ids"], s["counts"], FORMATS[s["case"]["fmt"]], s["out"])
        return s["out"]
    if do == "jump":
        mtgp.mtgp_jump(s["streams"], s["ids"], s["jumps"])
        mtgp.mtgp_generate_u32(s["streams"], s["ids"], s["counts"], s["out"])
        return s["out"]
    if do == "tests":
        hist = mtgp.mtgp_gap_histogram(s["values"], s["counts"], *GAP)
        table = mtgp.mtgp_hamming_pairs(s["values"], s["counts"], *HAMMING, s["bounds"])
        return [hist.view(np.int64), table.view(np.int64)]
    return _serve(s)


def work(case):
    """Each state read and written once, each number written once (read once
    per test); operations: 13 integer operations per number of MTGP, 15 of
    the original MT, 4 per number and test of the statistics."""
    if case["do"] == "jump":
        n = case["mexp"] // 32 + 1
        numbers = case["streams"] * case["draw"]
        # the jumped state: one window of the next Mexp words per state word
        return {"bytes": 4.0 * numbers + 16.0 * n * case["streams"], "flops": 13.0 * case["mexp"] * case["streams"]}
    numbers = float(_counts(case).sum())
    streams = case.get("streams") or case["requests"]
    if case["do"] == "tests":
        return {"bytes": 2 * 4.0 * numbers + 8.0 * streams * (GAP[2] + 1 + 16), "flops": 8.0 * numbers}
    n = (case["p"] + 31) // 32 if case["do"] == "mt" else case["mexp"] // 32 + 1
    b = 4.0 * numbers + 8.0 * n * streams
    if case["do"] == "stats":
        b += 8.0 * streams * (GAP[2] + 1 + 16)
    return {"bytes": b, "flops": (21.0 if case["do"] == "stats" else 15.0 if case["do"] == "mt" else 13.0) * numbers}


# ---------------------------------------------------------------------------
# The same numbers in plain numpy: the recurrences written out, advanced for
# all streams at once in blocks whose words do not depend on one another.
# ---------------------------------------------------------------------------
_M64 = (1 << 64) - 1


def _splitmix(seed):
    x = seed & _M64
    while True:
        x = (x + 0x9E3779B97F4A7C15) & _M64
        z = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & _M64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
        yield z ^ (z >> 31)


def _span(basis):
    return np.array([np.bitwise_xor.reduce([0] + [b for k, b in enumerate(basis) if i >> k & 1])
                     for i in range(16)], np.uint32)


def _plain_states(n, seeds):
    w = np.empty((seeds.size, n), np.uint32)
    w[:, 0] = seeds
    for i in range(1, n):
        p = w[:, i - 1]
        w[:, i] = np.uint32(1812433253) * (p ^ (p >> np.uint32(30))) + np.uint32(i)
    return w


def _plain_mtgp(mexp, pseed, seeds, most):
    """The first `most` outputs of every stream (streams x most words)."""
    d = _splitmix(int(pseed))
    n = mexp // 32 + 1
    sh1, sh2 = (np.uint32(1 + next(d) % 31) for _ in range(2))
    width = 1
    while width * 2 <= n - 2 and width < 256:
        width *= 2
    pos = 2 + next(d) % (n - width - 1)
    rec, tmp = (_span([next(d) >> 32 for _ in range(4)]) for _ in range(2))
    mask = np.uint32((0xFFFFFFFF << (32 * n - mexp)) & 0xFFFFFFFF)
    x = np.empty((seeds.size, n + most), np.uint32)
    x[:, :n] = _plain_states(n, seeds)
    out = np.empty((seeds.size, most), np.uint32)
    for i in range(0, most, n - pos):
        k = min(n - pos, most - i)
        y = (x[:, i:i + k] & mask) ^ x[:, i + 1:i + 1 + k]
        y ^= y << sh1
        y ^= x[:, i + pos:i + pos + k] >> sh2
        x[:, i + n:i + n + k] = y ^ rec[y & np.uint32(15)]
        t = x[:, i + pos - 1:i + pos - 1 + k]
        t = t ^ (t >> np.uint32(16))
        t ^= t >> np.uint32(8)
        out[:, i:i + k] = x[:, i + n:i + n + k] ^ tmp[t & np.uint32(15)]
    return out


def _plain_format(o, fmt):
    if fmt == "u32":
        return o.view(np.int32)
    return (o >> np.uint32(9)).astype(np.float64) * 2.0 ** -23 + (1.0 if fmt == "f32_12" else 0.0)


def exact(case, seed):
    """The numbers of the first pass; None for the large cases and for jumps,
    statistics and the comparison generator (whole numbers throughout)."""
    if case["do"] not in ("call", "plan", "serve") or case.get("sets"):
        return None
    counts = _counts(case).astype(np.int64)
    if int(counts.max()) * counts.size > 1 << 26:
        return None
    resident = case.get("resident", counts.size)
    ids = np.arange(counts.size) if case["do"] == "plan" else _ids(case, seed)
    o = _plain_mtgp(case["mexp"], workloads.PARAM_SEED, _seeds(resident, seed)[ids], int(counts.max()))
    if case["do"] == "serve":
        return [_plain_format(o[j, :k], "f32_01" if j % 2 else "u32") for j, k in enumerate(counts)]
    return np.concatenate([_plain_format(o[j, :k], case["fmt"]) for j, k in enumerate(counts)])
