"""The kernel without late tempering where it takes 128-word steps: many about
equal streams of a parameter set with N - pos < 256, and launches that a
CTA-wide phase takes whole; on both sides of the rule, against the oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 4


@pytest.mark.parametrize("entry", ["call", "plan"])
@pytest.mark.parametrize("mexp,gap,per_sm,coop,even,general", [
    (11213, 200, 13, 0, True, True),      # N - pos < 256, more streams than 12 per SM, equal
    (11213, 200, 13, 0, False, False),
    (11213, 200, 12, 0, True, False),
    (11213, 256, 13, 0, True, False),
    (23209, 140, 14, 0, True, True),
    (11213, 256, 8, 100, True, True),     # all of them CTA-wide
    (11213, 256, 9, 100, True, False),
    (11213, 256, 2, 100, True, False),
    (44497, 300, 7, 50, True, True)])
def test_many_even_streams(mexp, gap, per_sm, coop, even, general, entry):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, N = per_sm * sms + (0 if general or per_sm in (2, 8, 12) else 1), mexp // 32 + 1
    o0 = oracle.params_generate(mexp, 7)
    op = oracle.params_from_fields(mexp, N - gap, o0.sh1, o0.sh2, list(o0.rec_basis), list(o0.tmp_basis))
    p = mtgp.mtgp_params_create(mexp, N - gap, o0.sh1, o0.sh2, list(op.rec_tbl), list(op.tmp_tbl))
    seeds = np.arange(n, dtype=np.uint32)
    st = mtgp.mtgp_init_statuses(p, seeds)
    mtgp.mtgp_set_launch_config(st, warps_per_cta=4, ctas_per_sm=0, words_per_lane=4, kernel=0, coop_percent=coop)
    counts = np.full(n, 9 * N + 5, np.uint64)   # too long for the kernel of short streams
    counts[::7] -= 3
    if not even:
        counts[0] *= 4
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    out = torch.empty(int(counts.sum()), dtype=torch.int32, device="cuda")
    plan = mtgp.mtgp_plan_create(st, seeds, counts, mtgp.MTGP_F32_12, out) if entry == "plan" else None
    if plan:
        i = mtgp.mtgp_plan_get_info(plan)
        assert (i["resident_ctas_per_sm"] * 4 > (12 if mexp < 15000 else 8)) == general
        assert i["n_coop"] == (n if general and coop else 0) or not general
    for _ in range(2):
        if plan:
            mtgp.mtgp_plan_launch(plan)
        else:
            mtgp.mtgp_generate_f32(st, seeds, counts, mtgp.MTGP_F32_12, out)
        torch.cuda.synchronize()
        ref, states = oracle.generate_many(op, states, seeds, counts, mtgp.MTGP_F32_12, THREADS)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)
    mtgp.mtgp_check(st)
