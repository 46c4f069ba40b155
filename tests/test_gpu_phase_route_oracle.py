"""The one-step oracle tests of the sampled moments and tallies, through a
launch per phase.

Runs of their size take several steps per launch, so by themselves those tests
hold that route; large batches take the phase kernels, whose sample sums are
their own code.  The same tests with the same bounds on runs that take a launch
per phase (phase timing), and the sums of both routes with collisions.
"""
import numpy as np
import pytest

import helpers
import test_gpu_moments as moments
import test_gpu_parity as parity
import test_gpu_tallies as tallies
from paper_2308_13092_gb300 import inputs as I
from helpers import gpu_from_config, require_gpu
from test_gpu_several_steps import CASES

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


@pytest.fixture
def per_phase(monkeypatch):
    made = []

    def from_config(cfg, **kw):
        r = gpu_from_config(cfg, **kw)
        r.set_phase_timing(True)
        made.append(r)
        return r

    for m in (helpers, parity, tallies):
        monkeypatch.setattr(m, "gpu_from_config", from_config)
    yield
    assert made and all(r.route() is None for r in made)


@pytest.mark.parametrize("scheme,grid", [(I.EC, "uniform"), (I.EC, "doubling"), (I.MC, "uniform"),
                                         (I.MC, "doubling"), (I.EC2, "uniform"), (I.MC2, "uniform")])
def test_moments(per_phase, scheme, grid):
    moments.test_sample_step_moments_match_oracle_node_by_node(scheme, grid)


def test_moments_periodic_and_with_collisions(per_phase):
    moments.test_sample_step_moments_periodic()
    moments.test_sample_step_density_potential_energy_with_collisions()
    moments.test_density_of_quiet_neutral_cold_load_is_n0_on_the_gpu()


@pytest.mark.parametrize("scheme,grid,weights", [(I.EC, "uniform", False), (I.MC, "doubling", False),
                                                 (I.EC, "uniform", True), (I.EC2, "uniform", False)])
def test_moments_on_cell_sorted_particles(per_phase, scheme, grid, weights):
    moments.test_sample_step_moments_on_cell_sorted_particles(scheme, grid, weights)


@pytest.mark.parametrize("scheme,grid", [(I.EC, "uniform"), (I.MC, "uniform"), (I.EC2, "uniform"),
                                         (I.MC2, "uniform"), (I.EC, "tanh"), (I.MC, "tanh")])
def test_eedf_and_power(per_phase, scheme, grid):
    tallies.test_eedf_and_power_one_step(scheme, grid)


@pytest.mark.parametrize("scheme", [I.EC, I.MC, I.EC2, I.MC2])
def test_ion_impacts(per_phase, scheme):
    tallies.test_ion_impacts_one_step(scheme)


@pytest.mark.parametrize("case", [k for k in CASES if k not in ("one cell pair, few particles",
                                                                "no particle in a species")])
def test_sums_of_both_routes(case):
    """T_x, its averaged moments, J.E and the kinetic energy of one sample step
    of both routes, collisions included, node by node: each route's sums are
    within n + 8 roundings of 2^-24 of the terms (test_gpu_sample_sums.py, the
    launch per phase; collisions add FP64 changes of terms of the same size, at
    most one per particle), and T is a difference of two of them.  J.E's terms
    change sign; their sum of magnitudes is at most 2 |v|_rms E_max per particle
    over a cell (times 2 for the sampling of the speeds), and a particle may
    count in its old cell and stand in the next, or few cells on."""
    c = CASES[case]()
    c.sample_every = 33
    a, b = (gpu_from_config(c, sort_every=16) for _ in range(2))
    b.set_phase_timing(True)
    for r in (a, b):
        r.step(33)
        r.sync()
    assert a.route() is not None and b.route() is None
    da, db = a.diagnostics(), b.diagnostics()
    assert da["n_samples"] == db["n_samples"] == 1
    assert np.allclose(da["ke"], db["ke"], rtol=2e-6)
    N = a.N
    E = np.abs(b.fields()["E"]).max() * 1.5 + 1e-30
    for s, sp in enumerate(c.species):
        p = b.get_particles(s)
        k = b.get_weights(s) if getattr(c, "rebalance", None) else np.ones(p["cell"].size)
        n, M2, D = np.zeros(N + 1), np.zeros(N + 1), np.zeros(N + 1)
        f, v2 = p["xi"].astype(np.float64), p["vx"].astype(np.float64) ** 2
        for at, share in ((p["cell"], 1 - f), (p["cell"] + 1, f)):
            np.add.at(n, at, 1.0)
            np.add.at(M2, at, k * share * v2)
            np.add.at(D, at, k * share)
        if c.bc == I.PERIODIC:
            for x in (n, M2, D):
                x[0] += x[N]
                x[N] = x[0]
        ok = D > 0.5  # (a node with a sliver of a share has no temperature to speak of)
        tol = 8.0 * (2 * n + 8) * 2.0 ** -24 * sp.m / I.QE * M2 / np.maximum(D, 1e-30)
        for key in ("Tx", "Tx_mom"):
            off = np.abs(da[key][s] - db[key][s])
            assert np.all(off[ok] <= tol[ok]), (s, key, float(np.max(off[ok] / tol[ok])))
        vrms = np.sqrt((k * v2).sum() / max(k.sum(), 1.0))
        most = n.max() + 8
        scale = 0.5 * abs(sp.q) * sp.w * 4.0 * vrms * E / np.diff(c.edges) * max(D.max(), 1.0)
        off = np.abs(da["power"][s] - db["power"][s])
        assert np.all(off <= most * 2.0 ** -24 * scale), (s, float(np.max(off / scale)))
