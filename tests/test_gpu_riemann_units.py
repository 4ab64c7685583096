"""The exact Riemann solver in other units, and at the edges of its equations of state."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_16387_gb300 import workloads as WL

from test_gpu_parity import m2c  # noqa: F401

pytestmark = pytest.mark.gpu


def solve(M, eL, L, eR, R, **kw):
    import torch
    out, it, st = M.m2c_solve_riemann(eL, torch.from_numpy(L).cuda(), eR, torch.from_numpy(R).cuda(), **kw)
    return out.cpu().numpy(), st.cpu().numpy()


def mild_and_strong(n=3000):
    rng = np.random.default_rng(5)
    strong = rng.random(n) < 0.5
    L = np.stack([rng.uniform(980, 1150, n), rng.uniform(-150, 300, n),
                  np.where(strong, rng.uniform(1e8, 2e9, n), rng.uniform(9e4, 1e6, n))])
    R = np.stack([rng.uniform(0.8, 6.0, n), rng.uniform(-50, 50, n), rng.uniform(8e4, 5e6, n)])
    return L, R


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("k,m", [(-50, 0), (-34, -8), (40, 3)])
def test_mie_grueneisen_in_other_units(m2c, k, m, mixed):  # noqa: F811
    """Densities times 2^k, velocities times 2^m, pressures times 2^(k + 2m): the scaling is exact,
    and the result scales with it. Only the roots and reciprocals whose operands leave the seeds'
    range round differently; 1e-12 allows each of some thousand roundings of a curve one unit."""
    L, R = mild_and_strong()
    rho0, c0, s, g0 = WL.WATER_MG[1][:4]
    ref, rst = solve(m2c, WL.WATER_MG, L, WL.AIR_PG, R, mixed=mixed)
    scale = np.array([2.0 ** k, 2.0 ** m, 2.0 ** (k + 2 * m)])[:, None]
    water = (WL.WATER_MG[0], (rho0 * 2.0 ** k, c0 * 2.0 ** m, s, g0))
    out, st = solve(m2c, water, L * scale, WL.AIR_PG, R * scale, mixed=mixed)
    assert np.array_equal(st, rst) and (rst == 0).mean() > 0.99
    ok = rst == 0
    back = np.array([2.0 ** (k + 2 * m), 2.0 ** m, 2.0 ** k, 2.0 ** k])[:, None]
    for v in range(4):
        scale_v = np.maximum(np.abs(ref[v][ok]), 150.0 if v == 1 else 0.0)
        assert np.max(np.abs(out[v][ok] / back[v] - ref[v][ok]) / scale_v) < 1e-12, v


@pytest.mark.parametrize("water", [WL.WATER_SG, WL.WATER_MG], ids=["sg", "mg"])
def test_a_contact_keeps_its_states(m2c, water):  # noqa: F811
    """Equal pressures and velocities: no wave, and every value of the star states is its side's own."""
    n = 4000
    rng = np.random.default_rng(9)
    p, u = rng.uniform(8e4, 5e6, n), rng.uniform(-100, 100, n)
    L = np.stack([rng.uniform(990, 1100, n), u, p])
    R = np.stack([rng.uniform(0.8, 6.0, n), u, p])
    out, st = solve(m2c, water, L, WL.AIR_PG, R)
    assert (st == 0).all()
    assert np.array_equal(out, np.stack([p, u, L[0], R[0]]))


def wide(rng, lo, hi, n):
    """Wide states of a condensed material: a third in tension, velocities from 1 to 1e4."""
    p = np.where(rng.random(n) < 0.3, -rng.uniform(0, 3.6e8, n), np.exp(rng.uniform(np.log(1e3), np.log(1e10), n)))
    return np.stack([rng.uniform(lo, hi, n), rng.uniform(-1, 1, n) * 10 ** rng.uniform(0, 4, n), p])


def against_oracle(M, eL, L, eR, R):
    """Equal statuses; 1e-9 of each value (u*: of at least 1) where the oracle's Newton iteration
    converges. A problem that it leaves to the bisection has the jump of a curve at its root: the
    last bits decide which side of it is returned."""
    ref, rit, rst = O.riemann_batch(O.EOS(*eL), L, O.EOS(*eR), R)
    out, st = solve(M, eL, L, eR, R)
    assert np.array_equal(st, rst)
    ok = (rst == 0) & (rit <= 50)
    assert ok.sum() > 0.99 * (rst == 0).sum()
    for v in range(4):
        scale = np.maximum(np.abs(ref[v][ok]), 1.0 if v == 1 else 1e-300)
        assert np.max(np.abs(out[v][ok] - ref[v][ok]) / scale) < 1e-9, v


def test_roots_beyond_the_acoustic_bound(m2c):  # noqa: F811
    """Water against copper, both without a tension cutoff, down to tensions of 1e10 Pa, where the
    root can lie beyond the pressure span that the fixed nodes of the isentrope cover."""
    rng = np.random.default_rng(17)
    copper = (WL.WATER_MG[0], (8930.0, 3940.0, 1.489, 1.99))
    against_oracle(m2c, WL.WATER_MG, wide(rng, 900, 1500, 20000), copper, wide(rng, 8000, 11000, 20000))


@pytest.mark.parametrize("other", ["water", "air"])
def test_finite_tension_cutoff(m2c, other):  # noqa: F811
    """Water with a tension cutoff at a strain of -0.02: the same problems are refused, and the roots
    are the oracle's."""
    rng = np.random.default_rng(3)
    n = 20000
    water = (WL.WATER_MG[0], (1000.0, 1483.0, 1.75, 0.28, 0.0, -0.02))
    L = wide(rng, 800, 1500, n)
    if other == "water":
        against_oracle(m2c, water, L, water, wide(rng, 800, 1500, n))
    else:
        R = np.stack([np.exp(rng.uniform(np.log(0.01), np.log(100), n)), rng.uniform(-1, 1, n) * 10 ** rng.uniform(0, 4, n),
                      np.exp(rng.uniform(np.log(10), np.log(1e8), n))])
        against_oracle(m2c, water, L, WL.AIR_PG, R)
