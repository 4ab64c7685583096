"""Mixed-precision runs give the same bits from one version of the library to the next.

The digests in golden/mixed_bits.json are those of the library whose interface arithmetic
defined them (commit 4579b3f). A mixed grid rounds its FP64 interface states to binary32, so
that a change in their last bits can move a cell by 1e-7; nothing else looks at that. The
inputs use +, -, *, / and square roots only and are the same bits on every machine."""
import hashlib
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "mixed_bits.json")
SG, MG = (0, (6.12, 3.43e8)), (1, (1000.0, 1483.0, 1.75, 0.28))
AIR = (0, (1.4, 0.0))
CASES = {  # n, water, boundaries, options
    "mg_40x33x29": ((40, 33, 29), MG, (0,) * 6, None),
    "mg_67x24x41": ((67, 24, 41), MG, (0, 0, 1, 1, 0, 0), None),
    "mg_mirror_rk3_mc": ((35, 30, 27), MG, (2, 0, 2, 0, 2, 0), dict(rk=3, limiter=1)),
    "mg_llf": ((30, 34, 26), MG, (0,) * 6, dict(flux=1)),
    "mg_rz": ((70, 1, 90), MG, (2, 0, 0, 0, 0, 0), dict(geom=1, x0=0.0)),
    "sg_44x37x31": ((44, 37, 31), SG, (0,) * 6, None),
    "mg_fp32_start": ((33, 40, 28), MG, (0,) * 6, None),
}


def state(n, water, rz):
    """A bubble with the shock inside it: shocked water with waves, a wavy surface, squeezed gas."""
    h = 1.0 / max(n)
    z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) * h for k in n[::-1]], indexing="ij")
    size = [k * h for k in n]
    c = [0.5 * s for s in size]
    if rz:
        c[0], c[1] = 0.0, 0.5 * h
    wave = (x - c[0]) * (z - c[2]) * 3.0 - (y - c[1]) * (x + z) * 2.0 + 0.4 * (z - 0.3) * (z - 0.7)
    r = np.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)
    phi = r - 0.3 * min(s for s, k in zip(size, n) if k > 1) * (1.0 + 0.5 * wave)
    along, sa, v = (z, size[2], 3) if rz else (x, size[0], 1)
    behind = along < 0.5 * sa
    gas = phi < 0
    W = behind & ~gas
    G = behind & gas
    P = np.zeros((5,) + x.shape)
    P[0] = np.where(gas, np.where(G, 4.0, 1.2), np.where(W, 1200.0 + 60.0 * wave, 1000.0))
    P[v] = np.where(W, 500.0 * (1.0 + wave), np.where(G, 250.0 + 80.0 * wave, 0.0))
    P[1 if v == 3 else 3] = np.where(W, 30.0 * wave, 0.0)
    P[4] = np.where(gas, np.where(G, 1e6 * (1.0 + 0.3 * wave), 1e5), np.where(W, 8e8 * (1.0 + 0.3 * wave), 1e5))
    rho, p = P[0], P[4]

    def energy(eos):
        kind, prm = eos
        if kind == 0:
            return (p + prm[0] * prm[1]) / ((prm[0] - 1.0) * rho)
        eta = 1.0 - prm[0] / rho
        k0 = prm[0] * prm[1] * prm[1]
        pr = np.where(eta > 0, k0 * eta / ((1.0 - prm[2] * eta) * (1.0 - prm[2] * eta)), k0 * eta)
        return pr * eta / (2.0 * prm[0]) + (p - pr) / (prm[0] * prm[3])
    e = np.where(gas, energy(AIR), energy(water))
    ke = 0.5 * (P[1] * P[1] + P[2] * P[2] + P[3] * P[3])
    return h, np.stack([rho, rho * P[1], rho * P[2], rho * P[3], rho * (e + ke)]), phi


def digest(M, name):
    n, water, bc, opts = CASES[name]
    h, W, phi = state(n, water, n[1] == 1)
    g = M.Grid(n, h, bc, (water, AIR), precision=M.MIXED, options=opts)
    if name == "mg_fp32_start":
        g.set_riemann_start(True)
    g.set_state(W, phi)
    g.step(12)  # past the first reinitialisation
    g.sync()
    assert g.stats().interface_faces > 40
    s = hashlib.sha256()
    for t in (g.W, g.phi):  # (+ 0.0: a zero's sign does not count)
        s.update((t.cpu().numpy() + 0.0).tobytes())
    return s.hexdigest()


@pytest.mark.parametrize("name", list(CASES))
def test_mixed_run_repeats_its_bits(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2508_16387_gb300 import m2c as M
    with open(GOLDEN) as f:
        assert digest(M, name) == json.load(f)[name]
