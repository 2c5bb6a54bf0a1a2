"""Claims of more items than warps from one list (longest stream of at most
2^14 numbers) and from lists per SM (longer ones): every output and state
against the oracle on both sides of the rule, through direct calls, plans and
the allocation-free call."""
import os

import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 4


@pytest.mark.parametrize("entry", ["call", "plan", "noalloc"])
@pytest.mark.parametrize("longest", [40, 1 << 14, (1 << 14) + 1])
@pytest.mark.parametrize("mexp", [3217, 11213])
def test_both_sides_of_the_rule(mexp, longest, entry):
    n = 1000 if entry == "noalloc" else 3000
    p, op = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), oracle.params_generate(mexp, workloads.PARAM_SEED)
    seeds = np.arange(n, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses(p, seeds)
    if entry == "noalloc":   # fewer warps than items
        mtgp.mtgp_set_launch_config(st, warps_per_cta=2, ctas_per_sm=1, words_per_lane=2 if mexp == 3217 else 4,
                                    kernel=0, coop_percent=0)
    counts = (1 + (np.arange(n) * 7919) % min(longest, 900)).astype(np.uint64)
    counts[[3, n // 2]] = longest
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    out = torch.empty(int(counts.sum()), dtype=torch.int32, device="cuda")
    plan = mtgp.mtgp_plan_create(st, seeds, counts, mtgp.MTGP_U32, out) if entry == "plan" else None
    for _ in range(2):
        out.fill_(-1)
        if plan:
            mtgp.mtgp_plan_launch(plan)
        elif entry == "call":
            mtgp.mtgp_generate_u32(st, seeds, counts, out)
        else:
            mtgp.mtgp_generate_noalloc(st, seeds, counts, mtgp.MTGP_U32, out)
        torch.cuda.synchronize()
        ref, states = oracle.generate_many(op, states, seeds, counts, mtgp.MTGP_U32, THREADS)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
    mtgp.mtgp_check(st)
