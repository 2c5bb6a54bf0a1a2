"""The original MT's wide steps (W = n - m): counts around whole steps and
whole buffers of steps, for step widths of one to eight sub-steps, exactly and
not exactly filled, against the oracle."""
import os

import numpy as np
import pytest

import oracle.mt as omt
from paper_1501_07701_gb300 import mtgp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("p", [107, 521, 1023, 1279, 3217, 4423, 9689, 16383, 19937])
@pytest.mark.parametrize("fmt", [0, 2])
def test_wide_steps(p, fmt):
    q = mtgp.mtgp_mt_params_mt19937() if p == 19937 else mtgp.mtgp_mt_params_generate(p, 3)
    oq = omt.params_mt19937() if p == 19937 else omt.params_generate(p, 3)
    w, n = min(q.n - q.m, 256), q.n
    buf = max(2 * n + w, min(16 * n, 4096)) // w   # steps in about one buffer
    counts = [max(s * w + d, 1) for s in (0, 1, 2, 3, buf, buf + 1, 2 * buf) for d in (-1, 0, 1)]
    ids = np.concatenate([np.arange(len(counts)), np.arange(5)]).astype(np.uint32)
    counts = np.array(counts + [w, 2 * w, 7, 1, 3 * w + 1], np.uint64)
    mt = mtgp.mtgp_mt_init(q, np.arange(len(counts) - 5, dtype=np.uint32))
    states = np.stack([omt.init_state(oq, int(s)) for s in range(len(counts) - 5)])
    for _ in range(2):
        out = torch.zeros(int(counts.sum()), dtype=torch.int32, device="cuda")
        mtgp.mtgp_mt_generate(mt, ids, counts, fmt, out)
        torch.cuda.synchronize()
        ref, states = omt.generate_many(oq, states, ids, counts, fmt, os.cpu_count() or 4)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
    assert np.array_equal(mtgp.mtgp_mt_get_statuses(mt), states)
    mtgp.mtgp_mt_check(mt)
