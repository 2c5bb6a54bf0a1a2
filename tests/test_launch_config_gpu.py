"""Reading a handle's launch configuration and setting it again changes
nothing, and a configuration changed in one field does what it says."""
import numpy as np
import pytest

from paper_1501_07701_gb300 import mtgp, workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEFAULT_K = {3217: 2, 11213: 4, 44497: 4}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_07701_gb300 import build
    build.build()


def _handle(mexp, n=4096):
    return mtgp.mtgp_init_statuses(mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED), np.arange(n, dtype=np.uint32))


def _launches():
    """Counts of launches whose automatic shapes differ, by their number of
    items, the evenness of their lengths and the state size."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for n in (1, 4 * sms, 4 * sms + 40, 8 * sms, 9 * sms, 13 * sms, 20 * sms):
        out.append(np.full(n, 64, np.uint64))
        c = np.full(n, 64, np.uint64)
        c[0] = 5000                       # one stream far above a warp's share
        out.append(c)
    return out


def _shapes(st):
    out = []
    for c in _launches():
        buf = torch.empty(int(c.sum()), dtype=torch.int32, device="cuda")
        i = mtgp.mtgp_plan_get_info(mtgp.mtgp_plan_create(st, np.arange(c.size), c, mtgp.MTGP_U32, buf))
        out.append((i["config"]["warps_per_cta"], i["config"]["words_per_lane"], i["grid_ctas"],
                    i["resident_ctas_per_sm"], i["n_coop"]))
    return out


@pytest.mark.parametrize("mexp", sorted(DEFAULT_K))
def test_default_round_trip(mexp):
    fresh = _shapes(_handle(mexp))
    assert len(set(s[:1] + s[3:4] for s in fresh)) > 1     # the sizes do choose different shapes
    st = _handle(mexp)
    cfg = mtgp.mtgp_get_launch_config(st)
    assert cfg == dict(warps_per_cta=4, ctas_per_sm=2, words_per_lane=DEFAULT_K[mexp], kernel=0, coop_percent=0)
    mtgp.mtgp_set_launch_config(st, **cfg)
    assert mtgp.mtgp_get_launch_config(st) == cfg
    assert _shapes(st) == fresh
    # put back after another one, as a program does that tries shapes
    mtgp.mtgp_set_launch_config(st, **dict(cfg, warps_per_cta=8, ctas_per_sm=1))
    assert set(s[0] for s in _shapes(st)) == {8}
    mtgp.mtgp_set_launch_config(st, **cfg)
    assert _shapes(st) == fresh


def test_tuned_configuration_round_trip():
    st = _handle(11213)
    best = mtgp.mtgp_autotune(st, mtgp.MTGP_U32, 2048, 4096)
    assert mtgp.mtgp_get_launch_config(st) == best
    tuned = _shapes(st)
    mtgp.mtgp_set_launch_config(st, **dict(best, warps_per_cta=2, ctas_per_sm=1))
    mtgp.mtgp_set_launch_config(st, **best)
    assert _shapes(st) == tuned
    other = _handle(11213)
    mtgp.mtgp_set_launch_config(other, **best)
    assert _shapes(other) == tuned


@pytest.mark.parametrize("mexp", [11213, 44497])
def test_default_with_cta_wide_streams(mexp):
    st, twin = _handle(mexp, 64), _handle(mexp, 64)
    mtgp.mtgp_set_launch_config(st, **dict(mtgp.mtgp_get_launch_config(st), coop_percent=100))
    c = np.full(64, 500, np.uint64)
    c[3] = 60000
    out = [torch.empty(int(c.sum()), dtype=torch.int32, device="cuda") for _ in range(2)]
    plan = mtgp.mtgp_plan_create(st, np.arange(64), c, mtgp.MTGP_U32, out[0])
    i = mtgp.mtgp_plan_get_info(plan)
    assert i["n_coop"] > 0 and i["config"]["warps_per_cta"] == 4
    mtgp.mtgp_plan_launch(plan)
    mtgp.mtgp_generate_u32(twin, np.arange(64, dtype=np.uint32), c, out[1])
    torch.cuda.synchronize()
    assert torch.equal(*out)
    assert np.array_equal(mtgp.mtgp_get_statuses(st), mtgp.mtgp_get_statuses(twin))
