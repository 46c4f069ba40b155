"""Several steps per launch against a launch per phase.

A batch of moderate size advances several steps in one cooperative launch;
phase timing takes the same batch through a launch per kernel phase.  Both
run the same device code, so a run's particles, counters, density, potential
and fields are equal bit for bit over every form the launch accepts; the sums
added by FP64 atomics (T_x, power, KE) only agree to rounding (T_x of a single
launch's steps is held against the oracle node by node in test_gpu_moments.py).
"""
import numpy as np
import pytest

from paper_2308_13092_gb300 import inputs as I
from helpers import gpu_from_config, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _ccp(N, n, seed, **kw):
    c = I.ccp("s", N=N, n0=5e13, dt=1.0 / (400 * I.F_RF), ppc=0, v0=300.0, p_mtorr=kw.pop("p", 60.0), n_steps=0,
              seed=seed, L=kw.pop("L", 0.05), n_per_species=n, **kw)
    c.sample_every = 7
    return c


def _tanh(scheme, n=5003):
    return _ccp(0, n, 5, scheme=scheme, edges=I.tanh_edges(101, 0.05, 1e-4))


def _rebalanced(scheme, n=9001):
    c = _tanh(scheme, n)
    c.rebalance = dict(every=5, target=64, lo=40, hi=80, m0=16)
    return c


def _four():
    c = _ccp(150, 3001, 8)
    ion = c.species[1]
    c.species += [I.Species(q, 10 * ion.m, w * ion.w, ion.capacity, 2000, 0.1) for q, w in ((ion.q, 1.0), (-ion.q, 3.0))]
    return c


CASES = {
    "ec": lambda: _ccp(128, 8192, 1),
    "one cell pair, few particles": lambda: _ccp(2, 3, 2),
    "no particle in a species": lambda: _ccp(64, 1, 3),
    "mc, odd": lambda: _ccp(257, 10007, 4, scheme=I.MC),
    "ec2": lambda: _ccp(97, 6001, 5, scheme=I.EC2),
    "mc2": lambda: _ccp(97, 6001, 6, scheme=I.MC2),
    "tanh ec": lambda: _tanh(I.EC),
    "tanh mc": lambda: _tanh(I.MC),
    "high pressure": lambda: _ccp(300, 150001, 7, p=400.0),
    "four species": _four,
    "2048 cells": lambda: _ccp(2048, 100003, 9, L=0.3),
    "periodic": lambda: I.periodic_plasma(N=65, ppc=33, scheme=I.EC, ions=True, seed=3),
    "periodic mc2": lambda: I.periodic_plasma(N=65, ppc=33, scheme=I.MC2, ions=False, seed=4),
    "rebalanced ec": lambda: _rebalanced(I.EC),
    "rebalanced mc": lambda: _rebalanced(I.MC),
    # two particles per thread
    "ec, 60000": lambda: _ccp(128, 30001, 10),
    "ec2, 60000": lambda: _ccp(97, 30002, 11, scheme=I.EC2),
    "rebalanced ec, 60000": lambda: _rebalanced(I.EC, 30003),
    "rebalanced mc, 60000": lambda: _rebalanced(I.MC, 30003),
}


def _state(r):
    d = r.diagnostics()
    parts = []
    for s in range(r.ns):
        p = r.get_particles(s)
        o = np.argsort(p["id"], kind="stable")
        parts.append([p[k][o] for k in ("id", "cell", "xi", "vx", "vy", "vz")])
    return d, r.fields(), parts


@pytest.mark.parametrize("case", CASES)
def test_same_trajectory_as_a_launch_per_phase(case):
    a, b = (gpu_from_config(CASES[case](), sort_every=16) for _ in range(2))
    b.set_phase_timing(True)
    for n in (1, 16, 23):  # one step, up to a sort, across sorts
        a.step(n)
        b.step(n)
    a.sync()
    b.sync()
    (da, fa, pa), (db, fb, pb) = _state(a), _state(b)
    assert da["step"] == db["step"] == 40 and da["n_samples"] == db["n_samples"]
    assert da["species"] == db["species"]
    for k in ("phi", "E"):
        assert np.array_equal(fa[k], fb[k]), k
    for x, y in zip(pa, pb):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)
    for k in ("density", "eedf", "iedf", "iad"):
        assert np.array_equal(da[k], db[k]), k
    # FP64 prefix sums over another partition of the nodes
    assert np.allclose(da["phi"], db["phi"], rtol=0, atol=1e-12 * max(1.0, np.abs(db["phi"]).max()))
    assert np.allclose(da["ke"], db["ke"], rtol=2e-6) and np.isclose(da["fe"], db["fe"], rtol=1e-12)


def test_batch_of_different_runs():
    """Runs of one batch that end at their own steps, one without particles
    left to push, against each run alone through a launch per phase."""
    from paper_2308_13092_gb300 import ecpic
    cfgs = [CASES[k]() for k in ("ec", "mc, odd", "tanh ec", "ec2", "one cell pair, few particles", "high pressure")]
    ends = [40, 17, 33, 40, 5, 21]
    eng = ecpic.Engine(max_slots=8, max_cells=512, species_per_run=2)
    t = [eng.submit(c, n) for c, n in zip(cfgs, ends)]
    while sum(eng.pump(16)):
        pass
    for c, n, k in zip(cfgs, ends, t):
        d = eng.poll(k, diagnostics=True, profiles=True)["diag"]
        r = gpu_from_config(c)
        r.set_phase_timing(True)
        r.step(n)
        r.sync()
        e = r.diagnostics()
        assert d["step"] == e["step"] == n and d["species"] == e["species"]
        assert np.array_equal(d["density"], e["density"])
        assert np.allclose(d["phi"], e["phi"], rtol=0, atol=1e-12 * max(1.0, np.abs(e["phi"]).max()))


def test_runs_in_several_threads():
    """Runs of different sizes stepped from several threads, each on its own
    stream, against the same runs alone."""
    import threading
    cfgs = [_ccp(64 + 400 * k, 3000 * (k + 1), 20 + k) for k in range(5)]

    def advance(c, out, k):
        r = gpu_from_config(c)
        for _ in range(40):
            r.step(5)
        r.sync()
        out[k] = _state(r)[2]

    alone, at_once = [None] * 5, [None] * 5
    for k, c in enumerate(cfgs):
        advance(c, alone, k)
    t = [threading.Thread(target=advance, args=(c, at_once, k)) for k, c in enumerate(cfgs)]
    for x in t:
        x.start()
    for x in t:
        x.join()
    for a, b in zip(alone, at_once):
        assert b is not None
        for u, v in zip(a, b):
            assert all(np.array_equal(x, y) for x, y in zip(u, v))


def test_step_under_capture_is_refused():
    """A step counts levels on the host, so a caller's graph cannot hold it:
    the error leaves the run as it was."""
    import torch
    from paper_2308_13092_gb300 import ecpic
    s = torch.cuda.Stream()
    r, a = (ecpic.Run.from_config(CASES["ec"](), stream=s.cuda_stream) for _ in range(2))
    for x in (r, a):
        x.step(20)
        x.sync()
    with pytest.raises(Exception):
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s):
            r.step(1)
    for x in (r, a):
        x.step(20)
        x.sync()
    assert r.diagnostics()["step"] == 40
    for u, v in zip(_state(r)[2], _state(a)[2]):
        assert all(np.array_equal(x, y) for x, y in zip(u, v))
