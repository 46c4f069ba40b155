"""Loader against the oracle where its routes differ: velocities from pairs of
floats or, near the middle of two floats and for cold species, in FP64; cells by
guess (equal cells) or by search; quotients by reciprocal or by division.  The
floats are the rounded FP64 values: CUDA's and the C library's FP64 functions
differ by some 2^-51, which moves about one rounding in 2^26, so of at most 2e6
values two may differ, by one float."""
import numpy as np
import pytest

import oracle
from paper_2308_13092_gb300 import inputs as I
from helpers import gpu_from_config, oracle_from_config, require_gpu

pytestmark = pytest.mark.gpu


def _edges(kind):
    return {"doubling": lambda: oracle.doubling_grid(128, 0.05, 0.01, 1, 8),
            "tanh": lambda: I.tanh_edges(70, 0.05, 0.05 / 400)}.get(kind, lambda: None)()


@pytest.mark.parametrize("N,grid,n,quiet,T", [
    (2, "equal", 3, False, 2.0), (2, "equal", 1001, True, 2.0), (129, "equal", 100003, False, 2.0),
    (400, "equal", 300001, False, 1e-3), (400, "equal", 100001, True, 1e4), (2048, "equal", 50001, False, 300.0),
    (0, "doubling", 100003, False, 2.0), (0, "tanh", 100001, True, 2.0), (64, "equal", 5001, False, 0.0)])
def test_loader_rounds_as_fp64(N, grid, n, quiet, T):
    require_gpu()
    c = I.ccp("l", N=N, n0=5e13, dt=1.0 / (400 * I.F_RF), ppc=0, v0=300.0, p_mtorr=60.0, n_steps=0, seed=n + 7,
              L=0.05, n_per_species=n, edges=_edges(grid))
    c.quiet = quiet
    for sp in c.species:
        sp.T_eV = T
    g, o = gpu_from_config(c), oracle_from_config(c)
    for s in range(len(c.species)):
        p, q = g.get_particles(s), o.get_particles(s)
        oc, oxi = o.get_particles_cell(s)
        assert np.array_equal(p["cell"], oc)
        for got, want in [(p["xi"], np.minimum(oxi.astype(np.float32), np.float32(1 - 2.0 ** -24)))] + [
                (p[k], q[k].astype(np.float32)) for k in ("vx", "vy", "vz")]:
            off = got != want
            assert off.sum() <= 2
            assert np.all(np.abs(got[off].astype(np.float64) - want[off]) <= np.spacing(np.abs(want[off])))
