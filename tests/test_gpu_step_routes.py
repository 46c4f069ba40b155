"""Which way a run's steps are launched (ecpic_debug_route): several steps per
launch or a launch per phase."""
import pytest

from paper_2308_13092_gb300 import ecpic
from helpers import gpu_from_config, require_gpu
from test_gpu_several_steps import CASES, _ccp, _state

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("case", CASES)
def test_comparison_cases_take_both_routes(case):
    """The runs whose two routes are compared elsewhere do take them."""
    r = gpu_from_config(CASES[case](), sort_every=16)
    assert r.route() is None  # no step yet
    r.step(3)
    got = r.route()
    assert got and got["threads"] in (256, 512) and got["blocks"] == got["largest_team"] >= 1
    r.set_phase_timing(True)
    r.step(3)
    assert r.route() is None
    r.set_phase_timing(False)
    r.step(1)
    assert r.route() == got
    r.set_pass_grid(304)
    r.step(1)
    assert r.route() is None
    r.sync()


def test_engine_route():
    e = ecpic.Engine(max_slots=4, max_cells=256, species_per_run=2)
    for k in range(3):
        e.submit(_ccp(128, 4000 * (k + 1), k), 40)
    e.pump(20)
    got = e.route()
    assert got and got["blocks"] >= 3 and got["largest_team"] < got["blocks"]
    e.set_phase_timing(True)
    e.pump(10)
    assert e.route() is None


@pytest.mark.parametrize("n,parts,threads", [
    (600, 4, 256), (8192, 4, 256), (29127, 4, 512), (50000, 3, 512), (65536, 2, 512), (110000, 2, 512),
    (131072, 1, 512),
])
def test_a_small_run_leaves_room_for_others(n, parts, threads):
    """A block of several steps per launch has its SM to itself, so a run that
    cannot use them all takes a share, and runs on other streams the rest."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    r = gpu_from_config(_ccp(128, n, 3))
    r.step(2)
    got = r.route()
    assert got and got["threads"] == threads and got["blocks"] <= sms // parts, got
    if parts < 4:  # and no less than it needs
        assert got["blocks"] > sms // (parts + 1), got
    r.sync()


@pytest.mark.parametrize("million,several", [(2.0, True), (8.0, True), (20.0, False)])
def test_a_large_run_takes_a_launch_per_phase(million, several):
    """Beyond some 13 million particles of one run its blocks of several steps
    per launch have too few warps against the phase kernels'."""
    r = gpu_from_config(_ccp(1024, int(million * 5e5), 3, L=0.3))
    r.step(2)
    assert (r.route() is not None) == several
    r.sync()


def test_runs_at_their_end_hold_no_blocks():
    """A finished run that is still resident leaves its blocks to the others:
    here within one pump, whose steps go in chunks of at most 64."""
    e = ecpic.Engine(max_slots=2, max_cells=256, species_per_run=2)
    t = [e.submit(_ccp(128, 200000, 1), 200), e.submit(_ccp(128, 262144, 2), 10)]
    e.pump(5)
    both = e.route()
    assert both and both["largest_team"] < both["blocks"]
    e.pump(150)
    alone = e.route()
    assert alone and alone["largest_team"] == alone["blocks"] == both["blocks"]
    while sum(e.pump(64)):
        pass
    assert [e.poll(k, diagnostics=True)["diag"]["step"] for k in t] == [200, 10]


def test_a_run_filled_by_its_caller_gets_its_blocks():
    """Sizes follow set_particles: a run that starts with few particles and is
    filled afterwards gets the blocks of its new size."""
    import numpy as np
    c = _ccp(128, 64, 3)
    for s in c.species:
        s.capacity = 200000
    r = gpu_from_config(c)
    r.step(1)
    assert r.route()["blocks"] == 1
    n = 150000
    rng = np.random.default_rng(1)
    for s in range(2):
        v = rng.normal(0.0, 1e3, (3, n)).astype(np.float32)
        r.set_particles(s, rng.integers(0, 128, n), rng.random(n, np.float32) * np.float32(0.99), *v, np.arange(n))
    r.step(1)
    r.sync()
    assert r.route()["blocks"] >= 128 and r.route()["threads"] == 512


def test_refused_launch_takes_a_launch_per_phase():
    """More blocks than the device holds at once: the cooperative launch is
    refused on the host, nothing runs, and the steps go a launch per phase."""
    import numpy as np
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms >= 160:
        pytest.skip("a launch has at most 160 blocks")
    a, b = (gpu_from_config(_ccp(128, 150000, 3), sort_every=16) for _ in range(2))
    for r in (a, b):
        r.step(5)
        assert r.route()["blocks"] == sms
    a.debug_step_blocks(160)
    a.step(30)
    assert a.route() is None
    b.step(30)
    a.sync()
    b.sync()
    assert a.diagnostics()["species"] == b.diagnostics()["species"]
    for x, y in zip(_state(a)[2], _state(b)[2]):
        assert all(np.array_equal(u, v) for u, v in zip(x, y))
    a.debug_step_blocks(0)  # once refused, it stays a launch per phase
    a.step(1)
    assert a.route() is None
    a.sync()


def test_steps_past_the_end_of_every_run():
    """A pump for more steps than any run has left: nothing is launched for the
    rest, and the runs end as they do one pump at a time."""
    import numpy as np
    out = []
    for pumps in ((10, 400), (10, 10, 10, 10)):
        e = ecpic.Engine(max_slots=2, max_cells=256, species_per_run=2)
        t = [e.submit(_ccp(128, 4000, 1), 40), e.submit(_ccp(100, 3000, 2), 20)]
        for n in pumps:
            left = e.pump(n)
        assert left == (0, 0)
        out.append([e.poll(k, diagnostics=True, profiles=True)["diag"] for k in t])
    assert [d["step"] for d in out[0]] == [40, 20]
    for a, b in zip(*out):
        assert a["species"] == b["species"] and a["n_samples"] == b["n_samples"]
        assert np.array_equal(a["density"], b["density"])
