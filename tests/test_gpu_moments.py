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


# FP32 deviations with full mantissas, of one size and mixed over ten decades
# in a node, down to the smallest, and beside 1/2, where FP64 sums take over.
# A node's sums: n - 1 = 18 roundings of 2^-53 of the sum S of magnitudes at
# most, 2^-48 S with the two roundings that follow
@pytest.mark.parametrize("box", [(64, 5, 1), (41, 6, 5)])
@pytest.mark.parametrize("kind", ["mixed", "low", "half", 0.1, 1e-4, 1e-8, 1e-10, 1e-12, 1e-17, 1e-30, 1e-42])
def test_moments_of_full_mantissas(kind, box):
    nx, ny, nz = box
    Q = 9 if nz == 1 else 19
    g = np.random.default_rng(12)
    P = g.uniform(0.5, 1.0, (Q, nz, ny, nx)) * g.choice([-1.0, 1.0], (Q, nz, ny, nx))
    if kind == "mixed":
        P *= np.exp(g.uniform(math.log(1e-10), math.log(0.49), P.shape))
    elif kind == "low":
        P *= np.exp(g.uniform(math.log(1e-17), math.log(1e-7), P.shape))
    elif kind == "half":
        P *= 1e-3
        P[3, 0, 1, 2], P[5, 0, 2, 4] = np.nextafter(np.float32(0.5), np.float32(0)), -np.nextafter(np.float32(0.5), np.float32(0))
        P[4, 0, 3, 7], P[6, 0, 4, 9] = 0.5, -0.5
        P[7, 0, 1, 11], P[8, 0, 2, 13] = np.nextafter(np.float32(0.5), np.float32(1)), -0.75
    else:
        P *= kind
    P = P.astype(np.float32)
    sim = lbm.Sim(dict(lattice=Q, nx=nx, ny=ny, nz=nz, tau=0.8, force_model="e", storage="f32"),
                  inputs.empty_mask(nx, ny, nz), stage=False)
    buf = torch.zeros(sim.sizes[lbm.BUF_POP_A], dtype=torch.uint8, device="cuda")
    nxp = (nx + 63) // 64 * 64
    buf.view(torch.float32)[:Q * nz * ny * nxp].view(Q, nz, ny, nxp)[..., :nx] = torch.from_numpy(P).cuda()
    lbm.lbm_load_state(sim.ctx, buf, 1, sim.stream)
    e = velocities(Q)
    d = np.stack([np.roll(P[a].astype(np.float64), tuple(e[a][::-1]), axis=(0, 1, 2)) for a in range(Q)])
    S = np.abs(d).sum(0)
    node = lambda w: np.array([math.fsum(v) for v in (w[:, None] * d.reshape(Q, -1)).T]).reshape(S.shape)  # noqa: E731
    rho, j = 1.0 + node(np.ones(Q)), np.stack([node(e[:, k].astype(float)) for k in range(3)])
    v = j / rho
    v_ref = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device="cuda")
    change, total, _ = sim.residual(v_ref)
    got = v_ref.cpu().numpy()
    bound = 2.0 ** -48 * (S + np.abs(v) * (S + 1.0)) / np.abs(rho)
    assert np.all(np.abs(got - v) <= bound)
    speed = np.sqrt((v * v).sum(0))
    assert abs(total - math.fsum(speed.ravel())) <= math.fsum(np.sqrt((bound ** 2).sum(0)).ravel()) + 1e-13 * total
    assert change == total > 0
    mass, momentum, _ = sim.balance()
    assert abs(mass - math.fsum(rho.ravel())) <= 1e-13 * (rho.size + S.sum())
    for k in range(3):
        assert abs(momentum[k] - math.fsum(j[k].ravel())) <= 1e-13 * S.sum()
    sim.close()


# the residual's FP64 reciprocal (third-order iteration from FP32: 2^-13 of a
# unit in the last place before its rounding) and square root, one value at a
# time: v = j / rho with j a power of two is the reciprocal itself, and the sum
# over one node of |v| the root of v v; densities beyond FP32's range take the
# plain quotient and root
@pytest.mark.parametrize("exponent", [0, 60, -60, 125, -125, 300, -300])
def test_reciprocal_and_root_are_rounded(exponent):
    from fractions import Fraction
    unit = 2.0 ** exponent
    g = np.random.default_rng(7)
    nx, ny = 64, 8
    cfg = dict(lattice=9, ny=ny, nz=1, tau=0.8, rho0=unit, force_model="e", storage="f64")
    sim = lbm.Sim(dict(cfg, nx=nx), inputs.empty_mask(nx, ny, 1), stage=False)
    P = np.zeros((9, ny, nx))
    P[0] = (np.exp2(g.uniform(-5, 5, (ny, nx))) * g.uniform(1, 2, (ny, nx)) - 1.0) * unit
    P[1], P[3] = unit / 16, -unit / 16                       # j = (unit / 8, 0), no density
    lbm.lbm_load_state(sim.ctx, torch.from_numpy(P).cuda().view(torch.uint8), 1, sim.stream)
    v_ref = torch.zeros((3, 1, ny, nx), dtype=torch.float64, device="cuda")
    sim.residual(v_ref)
    v, rho = v_ref[0, 0].cpu().numpy(), P[0] + unit
    ulp = Fraction(1, 2) + Fraction(1, 2 ** 12)
    for got, r in zip(v.ravel(), rho.ravel()):
        assert abs(Fraction(got) - Fraction(unit) / 8 / Fraction(r)) <= ulp * Fraction(np.spacing(got))
    sim.close()
    sim = lbm.Sim(dict(cfg, nx=1, ny=1), inputs.empty_mask(1, 1, 1), stage=False)
    one = torch.zeros(sim.sizes[lbm.BUF_POP_A], dtype=torch.uint8, device="cuda")
    row = one.view(torch.float64)[:9 * 64].view(9, 64)
    v_ref = torch.zeros((3, 1, 1, 1), dtype=torch.float64, device="cuda")
    for d0, speed in list(zip(P[0].ravel(), v.ravel()))[:60]:
        row[0, 0], row[1, 0], row[3, 0] = d0, unit / 16, -unit / 16
        lbm.lbm_load_state(sim.ctx, one, 1, sim.stream)
        _, total, _ = sim.residual(v_ref, update=False)
        vv, err = speed * speed, ulp * Fraction(np.spacing(total))
        assert (Fraction(total) - err) ** 2 <= Fraction(vv) <= (Fraction(total) + err) ** 2
    sim.close()
