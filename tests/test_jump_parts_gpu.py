"""The jump kernel's residue accumulation: states after jumps against oracle
generation, for every number of CTAs that one jump is shared out over (it
depends on the number of jumps in a launch), every pass width, polynomials of
few and many words, and repeated and unsorted stream ids."""
import os

import numpy as np
import pytest

import oracle
from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
THREADS = os.cpu_count() or 4


def _check(mexp, n, jumps, ids=None, pseed=workloads.PARAM_SEED):
    p, op = mtgp.mtgp_params_generate(mexp, pseed), oracle.params_generate(mexp, pseed)
    seeds = np.arange(n, dtype=np.uint32) + 17
    st = mtgp.mtgp_init_statuses(p, seeds)
    states = np.stack([oracle.init_state(op, int(s)) for s in seeds])
    ids = np.arange(n, dtype=np.uint32) if ids is None else np.asarray(ids, np.uint32)
    jumps = np.broadcast_to(np.asarray(jumps, np.uint64), ids.shape)
    mtgp.mtgp_jump(st, ids, jumps)
    _, states = oracle.generate_many(op, states, ids, jumps, 0, THREADS)
    assert np.array_equal(mtgp.mtgp_get_statuses(st), states)


# 8, 4, 2 and 1 CTAs per jump on 152 SMs
@pytest.mark.parametrize("n", [1, 19, 20, 38, 40, 76, 77, 200])
def test_parts(n):
    _check(11213, n, 20011)


# one to four passes over the accumulator, each instantiation
@pytest.mark.parametrize("mexp", [107, 521, 3217, 4253, 9689, 11213, 19937, 23209, 44497])
@pytest.mark.parametrize("n", [3, 160])
def test_widths(mexp, n):
    _check(mexp, n, 30000 + np.arange(n) % 3)


# short polynomials: t^(J-1) itself while J - 1 is below the degree
@pytest.mark.parametrize("J", [1, 2, 31, 32, 33, 64, 511, 512, 513, 1024, 1025, 3000])
def test_low_degrees(J):
    _check(11213, 2, J)
    _check(3217, 2, J)


def test_ids_in_any_order():
    _check(11213, 6, [5, 700, 1, 0, 40000, 5, 9], [4, 1, 4, 0, 2, 1, 4])
