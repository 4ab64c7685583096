"""Mirror sides at both ends of axes shorter than a tile, against the oracle."""
import numpy as np
import pytest

from paper_2508_16387_gb300 import workloads as WL

from oracle import oracle as O
from test_gpu_symmetry_forms import both, m2c, rel_err  # noqa: F401

pytestmark = pytest.mark.gpu
S = 2


@pytest.mark.parametrize("n", [(2, 9, 5), (15, 2, 4), (16, 3, 7), (33, 2, 2), (7, 11, 3)])
def test_short_mirrored_axes_match_oracle(m2c, n):  # noqa: F811
    """FP64: 1e-11 for the residual and 1e-9 after six steps, as for the other mirror runs; mixed
    residual 5e-5 (about a dozen FP32 roundings of fluxes up to ten times the differences)."""
    bc = (S,) * 6
    z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in n[::-1]], indexing="ij")
    phi = x + 0.1 * y - 0.52
    P = np.zeros((5,) + x.shape)
    P[0] = np.where(phi < 0, 1000.0 + 20.0 * x, 1.2 + 0.2 * y)
    P[4] = np.where(phi < 0, 1e8 * (1.0 + 0.3 * x * y), 1e5 * (1.0 + 0.1 * z))
    P[1], P[2], P[3] = 20.0 * (0.5 - x), 10.0 * x * y, 5.0 * z
    eos = (WL.AIR_PG, WL.WATER_SG)
    g_or, ref, g, _ = both(m2c, n, 1.0 / max(n), bc, eos, P, phi, 6)
    assert max(rel_err(g.W.cpu().numpy(), ref.W)) <= 1e-9
    W0 = O.prims_to_cons(g_or, P, phi)
    R_ref, _, _ = O.residual(g_or, W0, phi)
    for prec, tol in ((0, 1e-11), (1, 5e-5)):
        g = m2c.Grid(n, 1.0 / max(n), bc, eos, precision=prec)
        g.set_prims(P, phi)
        R, _ = g.residual()
        g.sync()  # no state outside the grid was taken for a cell
        assert max(rel_err(R.cpu().numpy(), R_ref)) <= tol, prec
