"""Steps over partly uniform states (rows that copy their state, keep it, or leave out an axis beside
rows that do not), and interfaces of fewer, about as many and more faces than the schedulers'
lanes, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_16387_gb300 import workloads as WL

from test_gpu_bulk_rows import _partly_uniform
from test_gpu_parity import m2c, rel_err  # noqa: F401
from test_gpu_symmetry_forms import both

pytestmark = pytest.mark.gpu
S = 2


@pytest.mark.parametrize("water", [WL.WATER_SG, WL.WATER_MG], ids=["sg", "mg"])
@pytest.mark.parametrize("n,two_phase,bc,opts", [
    ((64, 9, 7), True, (0,) * 6, None), ((33, 17, 5), False, (1, 1, 0, 0, 1, 1), None),
    ((70, 19, 20), True, (0, 0, S, S, 0, 0), dict(rk=3, limiter=1)), ((40, 11, 9), True, (S, 0, 0, 0, 0, S), dict(rk=1))])
def test_steps_over_partly_uniform_states(m2c, n, two_phase, bc, opts, water):  # noqa: F811
    """FP64 1e-9 after eleven steps (a reinitialisation among them), as for the other runs; the
    residual is exactly zero where the oracle's is, in both precisions (a cell and its neighbours
    alike: every flux difference is of equal numbers)."""
    P, phi = _partly_uniform(n, two_phase)
    g_or, ref, g, _ = both(m2c, n, 1.0 / n[0], bc, (water, WL.AIR_PG), P, phi, 11, opts)
    assert max(rel_err(g.W.cpu().numpy(), ref.W)) <= 1e-9
    assert np.array_equal(g.phi.cpu().numpy() < 0, ref.phi < 0)
    R_ref, _, _ = O.residual(g_or, O.prims_to_cons(g_or, P, phi), phi)
    still = (R_ref == 0).all(axis=0) & (phi > 2.5 / n[0])  # (interface cells: FIVER's rounding)
    assert still.mean() > 0.15
    for prec in (0, 1):
        g = m2c.Grid(n, 1.0 / n[0], bc, (water, WL.AIR_PG), precision=prec, options=opts)
        g.set_prims(P, phi)
        R, _ = g.residual()
        assert (R.cpu().numpy()[:, still] == 0).all()


@pytest.mark.parametrize("ny,nz", [(3, 5), (24, 25), (26, 25), (140, 142)])
def test_interfaces_of_any_number_of_faces(m2c, ny, nz):  # noqa: F811
    """A plane interface of ny nz faces: 15, 600 and 650 on 608 schedulers, 19880 for 19456 lanes.
    FP64 residual 1e-11, as for random states."""
    n = (18, ny, nz)
    rng = np.random.default_rng(ny)
    P = np.zeros((5, nz, ny, 18))
    phi = np.broadcast_to((np.arange(18) - 2.6) / 18.0, (nz, ny, 18)).copy()
    air = phi < 0
    r = rng.uniform(-1, 1, (5, nz, ny, 18))
    P[0] = np.where(air, 1.2 + 0.3 * r[0], 1000.0 + 30.0 * r[0])
    P[1:4] = 20.0 * r[1:4]
    P[4] = np.where(air, 1e5 * (1 + 0.5 * r[4]), 1e8 * (1 + 0.5 * r[4]))
    eos = (WL.WATER_MG, WL.AIR_PG)
    g_or = O.Grid(n=n, h=1 / 18.0, eos=tuple(O.EOS(*e) for e in eos), bc=(0,) * 6)
    R_ref, _, _ = O.residual(g_or, O.prims_to_cons(g_or, P, phi), phi)
    g = m2c.Grid(n, 1 / 18.0, (0,) * 6, eos)
    g.set_prims(P, phi)
    R, _ = g.residual()
    g.sync()
    assert max(rel_err(R.cpu().numpy(), R_ref)) <= 1e-11
