"""Bulk kernel on partly uniform states (rows that leave out the face states and fluxes of an
axis beside rows that do not), at row, tile and chunk edges, and the Riemann solver on
batches from one problem to more than one warp per scheduler."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_16387_gb300 import workloads as WL

from test_gpu_parity import gpu_start, m2c, oracle_start, rel_err  # noqa: F401

pytestmark = pytest.mark.gpu


def _partly_uniform(n, two_phase):
    """Water at rest, air at rest beyond 3/4 of the x length, and single disturbed cells in the
    first and last row, column and plane and on both sides of the 32-cell and 8-row edges."""
    nx, ny, nz = n
    P = np.zeros((5, nz, ny, nx))
    phi = np.ones((nz, ny, nx))
    P[0], P[4] = 1000.0, 1e5
    if two_phase:
        x = np.arange(nx) + 0.5
        phi[:] = (0.75 * nx - x) / nx
        P[0][phi < 0] = 1.2
    for i, j, k in ((0, 0, 0), (31, 7, 1), (32, 8, 2), (16, ny - 1, nz - 1), (5, ny // 2, nz // 2)):
        c = (min(k, nz - 1), min(j, ny - 1), min(i, nx - 1))
        if phi[c] > 0:
            P[0][c], P[1][c], P[2][c], P[3][c], P[4][c] = 1040.0, 50.0, -30.0, 20.0, 1e8
    return P, phi


@pytest.mark.parametrize("water", [WL.WATER_SG, WL.WATER_MG], ids=["sg", "mg"])
@pytest.mark.parametrize("n,two_phase,bc", [((64, 9, 7), True, (0, 0, 0, 0, 0, 0)), ((33, 17, 5), False, (1, 1, 0, 0, 1, 1)),
                                            ((70, 3, 20), True, (0, 0, 1, 1, 0, 0)), ((32, 8, 4), False, (0, 0, 0, 0, 0, 0))])
def test_partly_uniform_residual_matches_oracle(m2c, n, two_phase, bc, water):  # noqa: F811
    """FP64 to rounding: fluxes of up to 4.4e8 against differences of 1e8, 1e-11 as for random
    states. Mixed: about a dozen FP32 roundings (6e-8 each) of fluxes up to 5 times the largest
    difference, 4e-6 expected, 5e-5 allowed; exactly zero where the FP64 residual is."""
    P, phi = _partly_uniform(n, two_phase)
    s = WL.Setup("rows", n, 1.0 / n[0], (water, WL.AIR_PG), bc, phi, np.zeros(phi.shape, np.uint8), {})
    g_or, W0 = oracle_start(s, P)
    R_ref, _, _ = O.residual(g_or, W0, phi)
    for prec, tol in ((0, 1e-11), (1, 5e-5)):
        for rows, tz in ((8, 0), (4, 1), (8, 3)):
            g = gpu_start(m2c, s, prec, prims=P)
            g.set_tiling(rows, tz)
            R, _ = g.residual()
            assert max(rel_err(R.cpu().numpy(), R_ref)) < tol, (prec, rows, tz)


@pytest.mark.parametrize("n", [1, 31, 33, 20001])
def test_riemann_batch_sizes(m2c, n):  # noqa: F811
    """Rounding-level agreement (1e-10, as for the fixed batch) for batches that fill a lane, a
    warp and every scheduler; half of the water states move away from the air (tension)."""
    import torch
    rng = np.random.default_rng(n)
    water = WL.WATER_MG
    L = np.stack([rng.uniform(985, 1150, n), rng.uniform(-150, 150, n), rng.uniform(1e5, 1e9, n)])
    R = np.stack([rng.uniform(0.5, 5.0, n), rng.uniform(-100, 100, n), rng.uniform(5e4, 5e6, n)])
    ref, _, rst = O.riemann_batch(O.EOS(*water), L, O.EOS(*WL.AIR_PG), R)
    for mixed in (False, True):
        out, _, st = m2c.m2c_solve_riemann(water, torch.from_numpy(L).cuda(), WL.AIR_PG, torch.from_numpy(R).cuda(),
                                           mixed=mixed)
        out, st = out.cpu().numpy(), st.cpu().numpy()
        assert np.array_equal(st, rst)
        ok = rst == 0
        for v in range(4):
            scale = np.maximum(np.abs(ref[v][ok]), 150.0 if v == 1 else 1e-300)  # u*: 1e-11 of water's sound speed
            assert ok.sum() == 0 or np.max(np.abs(out[v][ok] - ref[v][ok]) / scale) < 1e-10, (v, mixed)
