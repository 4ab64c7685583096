"""Interface faces that were at rest in the previous stage: their Newton iteration starts from a
star pressure within rounding of a side's own pressure."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_16387_gb300 import workloads as WL

from test_gpu_parity import m2c, rel_err  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p0", [1e5, 101325.0, 83000.0, 2.7e5, 7.3e4, 1.01e6])
def test_faces_leaving_rest_match_oracle(m2c, p0):  # noqa: F811
    """Water and air at rest at p0, a shock in the air that reaches the air cell of resting faces
    within the first step: FP64 1e-9 of the largest value as for the other runs. Mixed: a binary32
    strain is worth K0 2^-24 = 131 Pa, two of them a face pressure; three steps of dt/h <= 1.1e-4
    with two faces an axis move the momentum by 0.18, of 1000 at most: 2e-4. One face solved at
    its starting pressure is off by 5e-3 and more."""
    n = (38, 21, 19)
    h = 1.0 / max(n)
    z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) * h for k in n[::-1]], indexing="ij")
    size = [k * h for k in n]
    phi = np.sqrt((x - 0.5) ** 2 + (y - 0.5 * size[1]) ** 2 + (z - 0.5 * size[2]) ** 2) - 0.17
    gas, behind = phi < 0, x < 0.5
    P = np.zeros((5,) + x.shape)
    P[0] = np.where(gas, np.where(behind, 4.0, 1.2), 1000.0)
    P[1] = np.where(gas & behind, 250.0, 0.0)
    P[4] = np.where(gas & behind, 10.0 * p0, p0)
    eos, bc = (WL.WATER_MG, WL.AIR_PG), (0,) * 6
    g_or = O.Grid(n=n, h=h, eos=tuple(O.EOS(*e) for e in eos), bc=bc)
    ref = O.run(g_or, O.prims_to_cons(g_or, P, phi), phi, 3)
    for prec, tol in ((0, 1e-9), (1, 2e-4)):
        g = m2c.Grid(n, h, bc, eos, precision=prec)
        g.set_prims(P, phi)
        g.step(3)
        g.sync()
        assert max(rel_err(g.W.cpu().numpy(), ref.W)) <= tol, prec


def test_a_repeated_host_pass_repeats_its_result(m2c):  # noqa: F811
    """upload, ten steps, download three times on the same host state (the second time with another
    state in between): the faces' star pressures of an earlier pass only start the iteration. FP64
    1e-12 of the largest value: ten steps of a run whose roots agree to the iteration's tolerance."""
    import torch
    from test_gpu_mixed_bits import AIR, MG, state
    n = (45, 38, 33)
    h, W, phi = state(n, MG, False)
    g = m2c.Grid(n, h, (0,) * 6, (MG, AIR))
    g.set_state()
    W, phi = torch.from_numpy(W).contiguous().pin_memory(), torch.from_numpy(phi).contiguous().pin_memory()
    other = (W.flip(3).contiguous().pin_memory(), phi.flip(2).contiguous().pin_memory())
    other[0][1].neg_()
    out = []
    for src in ((W, phi), other, (W, phi)):
        res = (torch.empty_like(W).pin_memory(), torch.empty_like(phi).pin_memory())
        g.upload(*src)
        g.step(10)
        g.download(*res)
        g.sync()
        out.append(res[0].numpy())
    assert max(rel_err(out[2], out[0])) <= 1e-12
