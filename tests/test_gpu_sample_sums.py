"""Sampled sums (J.E, x temperatures, kinetic energy) of one sample step
against sums formed in FP64 from the particles before and after it, for the
launch per phase and for several steps per launch.

Collisionless periodic runs, so that the particles read back around the step
are the ones it summed.  The terms are the kernels' own FP32 values (shares
(1 - xi) v and xi v, J.E term (v + v') E); what is compared is the summation.
Bounds, with a = sum of |terms| at a node or cell, n its particles:

* launch per phase: FP32 partial sums per lane, warp and block, so at most
  n + 8 roundings of 2^-24 of a, with those of the second moments' products;
* several steps per launch: every term, a second moment's product included, is
  a float whose sums are exact in 48-bit fixed point, or FP64 where it lies
  outside that; so n 2^-53 + 2^-48 of a for the FP64 sums and T itself;
* the same with weight multipliers: pairs of floats, 2^-44 of a (2^-45 of
  the terms' sum of magnitudes per pair sum, a warp's and a lane's); the
  multiplier is a power of two, so it rounds nothing.

Kinetic energy: each term is rounded to FP32 once or twice (2^-24 of it, signs
at random), so 6 2^-24 a / sqrt(n) for six standard deviations and more; the
launch per phase rounds the four-term sums of a lane as well (3 more, of up to
4 terms: 4 times that).
"""
import numpy as np
import pytest

from paper_2308_13092_gb300 import inputs as I
from helpers import gpu_from_config, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    require_gpu()


def _run(N, ppc, scheme, steps, route, weights=False, fast=0.0, sort_every=16):
    """A run at the level before its first sample step: its particles, its
    field, then those after the step and its diagnostics."""
    c = I.periodic_plasma(N=N, ppc=ppc, scheme=scheme, ions=True, seed=11)
    c.sample_every = steps
    if weights:
        c.rebalance = dict(every=100000, target=64, lo=1, hi=2048, m0=4)
    r = gpu_from_config(c, sort_every=sort_every)
    if route == "phase":
        r.set_phase_timing(True)
    if steps > 1:
        r.step(steps - 1)
    if fast:  # one particle so fast that the others' squares are below the fixed point's range
        for s in range(r.ns):
            p = r.get_particles(s)
            p["vx"][3] = fast
            r.set_particles(s, *(p[k] for k in ("cell", "xi", "vx", "vy", "vz", "id")))
    r.sync()
    before = [r.get_particles(s) for s in range(r.ns)]
    E = r.fields()["E"].astype(np.float64)
    r.step(1)
    r.sync()
    after = [r.get_particles(s) for s in range(r.ns)]
    d = r.diagnostics()
    assert d["n_samples"] == 1
    return c, before, E, after, d


def _by_id(p):
    o = np.argsort(p["id"], kind="stable")
    return {k: p[k][o] for k in ("cell", "xi", "vx", "vy", "vz")}


def _at_nodes(N, c, t):
    out = np.zeros(N + 1)
    np.add.at(out, c, t[0])
    np.add.at(out, c + 1, t[1])
    out[0] += out[N]
    out[N] = out[0]
    return out


@pytest.mark.parametrize("route", ["phase", "several"])
@pytest.mark.parametrize("N,ppc,scheme,steps,weights,fast", [
    (64, 64, I.EC, 1, False, 0.0),       # one particle per thread, not yet in cell order
    (97, 301, I.EC, 20, False, 0.0),     # two
    (65, 900, I.MC, 20, False, 0.0),     # four, blocks of 256 threads
    (512, 513, I.EC, 20, False, 0.0),    # four, blocks of 512 threads
    (2048, 40, I.EC, 1, False, 0.0),     # more cells than the sums' window, and not in cell order
    (2048, 40, I.EC, 20, False, 0.0),
    (2048, 200, I.MC, 20, False, 0.0),
    (128, 200, I.EC2, 20, False, 0.0),
    (128, 150, I.EC, 20, False, 1e8),    # terms below the fixed point's range
    (2048, 40, I.EC, 20, False, 1e8),
    (97, 301, I.EC, 20, True, 0.0),      # weight multipliers
])
def test_sample_sums_against_fp64(route, N, ppc, scheme, steps, weights, fast):
    c, before, E, after, d = _run(N, ppc, scheme, steps, route, weights, fast)
    f32 = np.float32
    dx = np.diff(c.edges)
    for s, sp in enumerate(c.species):
        p, q = _by_id(before[s]), _by_id(after[s])
        assert p["cell"].size == q["cell"].size
        cell, f, v = q["cell"], q["xi"], q["vx"]
        # the deposit, in integers; the quadratic one from the density, known to
        # the rounding of the node positions
        r = np.floor(f.astype(np.float64) * 2.0 ** 32)
        D, dD = _at_nodes(N, cell, (2.0 ** 32 - r, r)) * 2.0 ** -32, 0.0
        if scheme == I.EC2:
            D, dD = d["density"][s] * dx.mean() / sp.w, 2.0 * (dx.max() / dx.min() - 1.0)
        num = _at_nodes(N, cell, (np.ones(v.size), np.ones(v.size)))
        lo, hi = (f32(1) - f) * v, f * v
        assert lo.dtype == hi.dtype == f32
        lo, hi, v64 = lo.astype(np.float64), hi.astype(np.float64), v.astype(np.float64)
        M1 = _at_nodes(N, cell, (lo, hi))
        pl, ph = lo * v64, hi * v64
        if route == "several" and not weights:
            pl, ph = pl.astype(f32).astype(np.float64), ph.astype(f32).astype(np.float64)
        M2 = _at_nodes(N, cell, (pl, ph))
        A1 = _at_nodes(N, cell, (np.abs(lo), np.abs(hi)))
        T = sp.m * (M2 / D - (M1 / D) ** 2) / I.QE
        if route == "phase":
            d1, d2 = (num + 8) * 2.0 ** -24 * A1, (num + 8) * 2.0 ** -24 * M2
        elif weights:
            d1, d2 = 2.0 ** -44 * A1, 2.0 ** -44 * M2
        else:
            d1, d2 = 0.0 * A1, 0.0 * M2
        d1, d2 = d1 + (num * 2.0 ** -53 + 2.0 ** -48) * A1, d2 + (num * 2.0 ** -53 + 2.0 ** -48) * M2
        tol = sp.m / I.QE * (d2 / D + 2.0 * np.abs(M1) / D ** 2 * d1 + (d1 / D) ** 2 + (2.0 ** -48 + 3.0 * dD) * M2 / D)
        for key in ("Tx", "Tx_mom"):
            off = np.abs(d[key][s] - T)
            assert np.all(off <= tol), (s, key, float(np.max(off / tol)))
        # kinetic energy
        a = p["vx"].astype(np.float64) * q["vx"] + p["vy"].astype(np.float64) ** 2 + p["vz"].astype(np.float64) ** 2
        ke = 0.5 * sp.m * sp.w * a.sum()
        if fast == 0.0:
            off = abs(d["ke"][s] / ke - 1.0)
            assert off <= (24.0 if route == "phase" else 6.0) * 2.0 ** -24 / np.sqrt(a.size), (s, off)
        if scheme == I.EC:
            t = ((p["vx"] + q["vx"]) * E[p["cell"]].astype(f32)).astype(np.float64)
            P, A = np.zeros(N), np.zeros(N)
            np.add.at(P, p["cell"], t)
            np.add.at(A, p["cell"], np.abs(t))
            n = np.bincount(p["cell"], minlength=N)
            scale = 0.5 * sp.q * sp.w / dx
            eps = (n + 8) * 2.0 ** -24 if route == "phase" else 2.0 ** -44 if weights else 0.0
            tol = np.abs(scale) * (eps + n * 2.0 ** -53 + 2.0 ** -48) * A
            off = np.abs(d["power"][s] - scale * P)
            assert np.all(off <= tol), (s, float(np.max(off / np.maximum(tol, 1e-300))))
