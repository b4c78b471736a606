"""The FP64 reductions over nodes (balance, steady residual) against correctly
rounded host sums of the exported populations, where the exact integer sums of
FP32 deviations change to FP64 sums (a deviation of 1/2 or more), on boxes
smaller than a warp, of less than a block per SM and with closed faces and
solids."""
import math

import numpy as np
import pytest
import torch

from paper_2512_12213_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def velocities(Q):
    e = [(0, 0, 0)]
    if Q == 9:
        return np.array(e + [(1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)])
    for v in [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]:
        e += [v, tuple(-c for c in v)]
    return np.array(e)


# the values are exact in each format (seven bits).
# Sums: 1e-13 of the sum of magnitudes (n 2^-53 for n < 1e3 additions of a
# thread and block); velocities: a division and few roundings each
@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("box,scale", [((5, 3, 1), 1 / 16), ((67, 41, 1), 1 / 4), ((33, 9, 7), 1 / 16), ((70, 40, 30), 1 / 2),
                                       ((70, 40, 30), 1.0)])
def test_balance_and_residual_sums(box, scale, storage):
    nx, ny, nz = box
    Q = 9 if nz == 1 else 19
    mask = inputs.random_solids(nx, ny, nz, 0.1, seed=4)
    mask[nz // 2, ny // 2, nx // 2] = 0
    cfg = dict(lattice=Q, nx=nx, ny=ny, nz=nz, periodic=(1, 0, 1), tau=0.8, force_model="e", g=(2.0 ** -10, 0, 0),
               storage=storage, wall_u=((0, 0, 0),))
    sim = lbm.Sim(cfg, mask, stage=False)
    g = np.random.default_rng(8)
    d = np.round(g.uniform(-1, 1, (Q, nz, ny, nx)) * 64) / 64 * scale / 8
    d[0, nz // 2, ny // 2, nx // 2] = scale               # one node with a large deviation
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if Q == 9 else [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    f = d + w[:, None, None, None]
    sim.import_f(torch.from_numpy(f).cuda())
    e, fluid = velocities(Q), mask == 0
    rho = 1.0 + d.sum(0)
    j = np.tensordot(e.T, d, 1)
    mass, momentum, force = sim.balance()
    tiny = 1e-13 if storage == "f64" else 0.0              # FP64 stores f - w with w's rounding
    assert abs(mass - math.fsum(rho[fluid])) <= (1e-13 + tiny) * fluid.sum()
    for k in range(3):
        assert abs(momentum[k] - math.fsum(j[k][fluid])) <= (1e-13 + tiny) * np.abs(d).sum()
    assert abs(force[0] - 2.0 ** -10 * math.fsum(rho[fluid])) <= (1e-13 + tiny) * fluid.sum()
    v_ref = torch.full((3, nz, ny, nx), 0.25, dtype=torch.float64, device="cuda")
    if not np.all(rho[fluid]):                             # a node without mass has no velocity
        with pytest.raises(lbm.LbmError) as e:
            sim.residual(v_ref)
        assert e.value.status == lbm.ERR_NAN
        return
    v = j / rho
    v[0] += 2.0 ** -11
    change, total, _ = sim.residual(v_ref)
    assert abs(total - math.fsum(np.sqrt((v * v).sum(0))[fluid])) <= 1e-12 * fluid.sum()
    assert abs(change - math.fsum(np.sqrt(((v - 0.25) ** 2).sum(0))[fluid])) <= 1e-12 * fluid.sum()
    assert np.abs(v_ref.cpu().numpy() - np.where(fluid, v, 0.0)).max() <= 1e-13
    sim.close()
