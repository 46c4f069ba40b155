"""Several steps per launch across its sorts, bit for bit against a launch per
phase: a sort after every step or every second one, samples on every step,
births in every step (hot electrons: an ion and an electron enter the buffer
set that the sort has just left behind or filled), a rebalancing at the level
of a sort, and launches long enough for every rotation inside them (the
electrode's next 32 potentials, the counters' flush).
"""
import numpy as np
import pytest

from paper_2308_13092_gb300 import inputs as I
from helpers import gpu_from_config, require_gpu
from test_gpu_several_steps import _state

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _ionising(n, sample_every, scheme=I.EC, grid="uniform", rb=0):
    edges = I.tanh_edges(101, 0.05, 1e-4) if grid == "tanh" else None
    c = I.ccp("s", N=128, n0=5e13, dt=1.0 / (400 * I.F_RF), ppc=0, v0=300.0, p_mtorr=800.0, n_steps=0, seed=17,
              L=0.05, n_per_species=n, scheme=scheme, edges=edges, Te=40.0, headroom=4.0)
    c.sample_every = sample_every
    if rb:
        c.rebalance = dict(every=rb, target=64, lo=40, hi=80, m0=16)
    return c


@pytest.mark.parametrize("n,sort_every,sample_every,scheme,grid,rb", [
    (4099, 1, 1, I.EC, "uniform", 0),     # a few blocks
    (8192, 1, 7, I.EC, "uniform", 0),
    (30001, 2, 1, I.MC, "uniform", 0),
    (30001, 3, 2, I.EC, "tanh", 0),
    (30001, 1, 0, I.EC2, "uniform", 0),
    (150001, 1, 3, I.EC, "uniform", 0),   # blocks of 512 threads
    (9001, 5, 5, I.EC, "tanh", 5),        # sample, sort and rebalancing at one level
    (9001, 1, 1, I.MC, "tanh", 2),
    (30003, 4, 3, I.EC, "tanh", 2),
])
def test_births_across_sorts(n, sort_every, sample_every, scheme, grid, rb):
    a, b = (gpu_from_config(_ionising(n, sample_every, scheme, grid, rb), sort_every=sort_every) for _ in range(2))
    b.set_phase_timing(True)
    for m in (1, 99, 20):
        a.step(m)
        b.step(m)
    a.sync()
    b.sync()
    (da, fa, pa), (db, fb, pb) = _state(a), _state(b)
    births = db["species"][0]["births"]
    assert births > 120, births  # more than one per step
    assert da["step"] == db["step"] == 120 and da["n_samples"] == db["n_samples"]
    assert da["species"] == db["species"]
    for k in ("phi", "E"):
        assert np.array_equal(fa[k], fb[k]), k
    for x, y in zip(pa, pb):
        assert np.unique(x[0]).size == x[0].size  # no particle twice
        for u, v in zip(x, y):
            assert np.array_equal(u, v)
    for k in ("density", "eedf", "iedf", "iad"):
        assert np.array_equal(da[k], db[k]), k
    if sample_every:
        assert np.allclose(da["phi"], db["phi"], rtol=0, atol=1e-12 * max(1.0, np.abs(db["phi"]).max()))
